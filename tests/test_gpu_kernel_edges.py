"""Kernels at the sizes where their work split changes: remainders, tile edges, the smallest and
largest of a range, against the oracle or a plain NumPy statement of the same arithmetic."""
import numpy as np
import pytest

import synth
from oracle import classify as OC
from oracle import forces as OF
from oracle.grid import Grid
from tests.gpu_util import assert_tables_equal, classify_both, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    import paper_2605_04335_gb300 as pkg
    c = pkg.Context(0)
    yield pkg, c
    c.close()


def _double_cone(n):
    """Closed body of 2 n triangles whose two apexes have n triangles each; one vertex unused."""
    a = 2.0 * np.pi * np.arange(n) / n
    ring = np.stack([0.5 + 0.23 * np.cos(a), 0.5 + 0.23 * np.sin(a), np.full(n, 0.49)], 1)
    v = np.concatenate([ring, [[0.51, 0.5, 0.74], [0.9, 0.9, 0.9], [0.5, 0.48, 0.27]]])
    i = np.arange(n)
    j = (i + 1) % n
    t = np.concatenate([np.stack([i, j, np.full(n, n)], 1), np.stack([j, i, np.full(n, n + 2)], 1)])
    return synth.Mesh(v, t[np.random.RandomState(n).permutation(2 * n)].astype(np.int32), 1)


@pytest.mark.parametrize("n", [3, 31, 32, 33, 64, 65, 200])
def test_nodal_forces_by_valence(ctx, n):
    """Nodes of n triangles (a warp holds 32 at once): bit for bit the oracle's ordered sums."""
    pkg, c = ctx
    f = synth.faces_uniform(24)
    grid = Grid(f, f, f)
    m = _double_cone(n)
    ib = OC.iblank_closed(grid, [m])
    p = synth.counter_normal(5, 0, np.arange(24 ** 3)).reshape(grid.shape)
    T = pkg.Tables(c, f, f, f, [m])
    out = T.surface_forces([m], torch.from_numpy(p).cuda())
    ps, _, F = OF.surface_forces(grid, ib, [m], p)
    assert np.array_equal(out["p_side"].cpu().numpy(), ps)
    assert np.array_equal(out["f_node"].cpu().numpy(), F)
    T.close()


@pytest.mark.parametrize("n", [3, 511, 512, 513, 1024, 1025])
def test_classification_by_triangle_count(ctx, n):
    """2 n triangles (the scans run 1024 counts at a time): tables bit for bit the oracle's."""
    pkg, c = ctx
    f = synth.faces_uniform(24)
    _, T, ex, ib, G = classify_both(pkg, c, f, f, f, [_double_cone(n)])
    assert_tables_equal(ex, ib, G)
    T.close()


@pytest.mark.parametrize("shape", [(64, 64, 1023), (64, 64, 1024), (67, 64, 1024), (129, 131, 260)])
def test_ghost_compaction_by_grid_size(ctx, shape):
    """Ghost lists of grids around 1024 blocks of the compaction (4096 cells each)."""
    pkg, c = ctx
    xf, yf, zf = [synth.faces_uniform(n) for n in shape]
    _, T, ex, ib, _ = classify_both(pkg, c, xf, yf, zf, [synth.octa_sphere(3, (0.5, 0.5, 0.5), 0.41)], oracle_ghosts=False)
    assert np.array_equal(ex["iblank"], ib)
    assert np.array_equal(ex["cell"], np.flatnonzero(ib.ravel() == 3))
    T.close()


@pytest.mark.parametrize("case", ["cone", "fine_mesh", "coarse_mesh", "far_coordinates", "tiny_triangles", "boxes"])
def test_closest_triangle_search(ctx, case):
    """Boundary intercepts bit for bit the oracle's: slivers, many triangles per cell, many cells
    per triangle, coordinates near the limit of 4, edges below the FP32 bounds' range, flat faces
    with equally near triangles."""
    pkg, c = ctx
    n, lo, hi = 24, 0.0, 1.0
    if case == "cone":
        meshes = [_double_cone(150)]
    elif case == "fine_mesh":
        n, meshes = 14, [synth.octa_sphere(5, (0.5, 0.49, 0.51), 0.3)]
    elif case == "coarse_mesh":
        n, meshes = 40, [synth.octa_sphere(0, (0.5, 0.49, 0.51), 0.33)]
    elif case == "far_coordinates":
        lo, hi = 3.0, 4.0
        meshes = [synth.ellipsoid(4, (0.2, 0.11, 0.08), 20.0, (3.52, 3.48, 3.51))]
    elif case == "tiny_triangles":
        lo, hi = 0.5, 0.504
        meshes = [synth.octa_sphere(5, (0.50203, 0.50198, 0.50201), 0.0011)]
    else:
        meshes = [synth.box_mesh((0.1, 0.1, 0.1), (0.4, 0.45, 0.9)), synth.octa_sphere(3, (0.7, 0.5, 0.5), 0.17)]
    f = lo + (hi - lo) * synth.faces_uniform(n)
    _, T, ex, ib, G = classify_both(pkg, c, f, f, f, meshes)
    assert len(G) > 20
    assert_tables_equal(ex, ib, G)
    T.close()


@pytest.mark.parametrize("shape", [(33, 18, 21), (34, 19, 20), (35, 17, 18), (65, 31, 40), (130, 12, 15), (24, 9, 70)])
def test_solves_at_odd_sizes(ctx, shape):
    """Every precision against the oracle's direct solve: rows of 1, 2 and 3 cells beyond a strip,
    odd and even planes, long and short rows on the coarse levels."""
    from oracle import solve as OS
    pkg, c = ctx
    n = max(shape)
    f = [m / n * synth.faces_tanh(m, 1.5) for m in shape]
    size = min(shape) / n
    mid = [0.5 * m / n for m in shape]
    mesh = synth.ellipsoid(3, (0.33 * size, 0.26 * size, 0.29 * size), 25.0, mid)
    g, T, _, ib, G = classify_both(pkg, c, *f, [mesh])
    b = synth.rhs_divergence(*f, 3)
    p_o, _ = OS.solve_sparse(g, ib, G, b)
    fl = ib == 0
    for prec in (0, 1, 2):
        p = torch.zeros(b.shape, dtype=torch.float64, device="cuda")
        T.solve(torch.from_numpy(b).cuda(), p, 1e-11, pkg.SolveOpts(precision=prec))
        err = np.linalg.norm((p.cpu().numpy() - p_o)[fl]) / np.linalg.norm(p_o[fl])
        assert err < 1e-8, (prec, err)
    T.close()


@pytest.mark.parametrize("shape", [(2, 2, 2), (31, 3, 16), (32, 5, 17), (33, 2, 15), (62, 4, 33), (63, 7, 32), (100, 9, 40)])
def test_noalloc_residual_at_march_edges(ctx, shape):
    """The allocation-free residual (marches of 16 planes, 31 or 32 cells along x) against the oracle's,
    with a large mean in p and in the right-hand side; p undefined (NaN) inside the body."""
    from oracle import system as OY
    pkg, c = ctx
    f = [synth.faces_tanh(m, 1.7) for m in shape]
    big = min(shape) > 8
    meshes = [synth.octa_sphere(2, (0.5, 0.5, 0.5), 0.3)] if big else []
    g, T, ex, ib, G = classify_both(pkg, c, *f, meshes)
    e = T.export()
    b = synth.counter_normal(3, 0, np.arange(ib.size)).reshape(ib.shape) + 5.0
    p = synth.smooth_field(*f, 4) + 1e-3 * synth.counter_normal(3, 1, np.arange(ib.size)).reshape(ib.shape)
    p_nan = np.where(ib == 1, np.nan, p)
    rel, sr, sb = pkg.ibm_residual_norm_noalloc(*f, e["iblank"], e["cell"], e["ref"], e["w"], e["scale"],
                                                torch.from_numpy(b).cuda(), torch.from_numpy(p_nan).cuda())
    rf, rg = OY.residual(g, ib, G, b, p, 0.0)
    want = OY.projected_norm(g, ib, G, rf, rg)
    base = OY.projected_norm(g, ib, G, np.where(ib == 0, b, 0.0), np.zeros(len(G)))
    # a residual cell carries about 10 roundings of sum |c| |p| and of the mean of b
    assert abs(sr - want) <= 1e-12 * want and abs(sb - base) <= 1e-12 * base and abs(rel - want / base) <= 2e-12 * rel
    T.close()


@pytest.mark.parametrize("shape", [(33, 18, 21), (34, 19, 20), (35, 17, 18), (64, 16, 32), (130, 13, 15), (9, 24, 70)])
def test_velocity_solve_at_odd_sizes(ctx, shape):
    """The FP32 strip sweep (4 cells, 2 planes), the marched double-FP32 residual and the packs of 4 rows
    against the oracle's direct solve; a second solve starts from correction arrays in use."""
    from oracle import helmholtz as OH
    pkg, c = ctx
    n = max(shape)
    f = [m / n * synth.faces_tanh(m, 1.5) for m in shape]
    size = min(shape) / n
    mesh = synth.ellipsoid(3, (0.33 * size, 0.26 * size, 0.29 * size), 25.0, [0.5 * m / n for m in shape])
    g, T, _, ib, G = classify_both(pkg, c, *f, [mesh])
    S = (np.max(g.cxm + g.cxp) + np.max(g.cym + g.cyp)) + np.max(g.czm + g.czp)
    rhs = synth.smooth_field(*f, 3) + 0.1 * synth.counter_normal(6, 0, np.arange(ib.size)).reshape(ib.shape)
    ub = synth.counter_normal(7, 0, np.arange(len(G)))
    fd, ubd = torch.from_numpy(rhs).cuda(), torch.from_numpy(ub).cuda()
    for aS in (0.7, 2.5):
        u_o = OH.solve_closed(g, ib, G, aS / S, rhs, ub)
        for prec in (0, 1, 2):
            u = torch.zeros_like(fd)
            rep = T.helmholtz_solve(aS / S, fd, u, ubd, 1e-11, pkg.HelmholtzOpts(precision=prec))
            got = u.cpu().numpy()
            err = np.linalg.norm((got - u_o)[ib != 1]) / np.linalg.norm(u_o[ib != 1])
            assert rep["status"] == "IBM_OK" and err <= 1e-8, (aS, prec, err)
            assert np.all(got[ib == 1] == 0.0)
    T.close()


@pytest.mark.parametrize("shape", [(32, 32, 32), (33, 32, 31), (34, 32, 32), (16, 16, 16), (130, 40, 9), (12, 9, 150), (20, 24, 17)])
def test_coarse_tail_edges(ctx, shape):
    """The one-block coarse tail at its largest level (16^3 cells), just past it, at the corner-by-corner
    limit (8^3) and on long levels: every precision against the oracle's direct solve."""
    from oracle import solve as OS
    pkg, c = ctx
    n = max(shape)
    f = [m / n * synth.faces_tanh(m, 1.4) for m in shape]
    size = min(shape) / n
    mesh = synth.ellipsoid(3, (0.31 * size, 0.27 * size, 0.24 * size), 25.0, [0.5 * m / n for m in shape])
    g, T, _, ib, G = classify_both(pkg, c, *f, [mesh])
    b = synth.rhs_divergence(*f, 3)
    p_o, _ = OS.solve_sparse(g, ib, G, b)
    fl = ib == 0
    for prec in (0, 1, 2):
        p = torch.zeros(b.shape, dtype=torch.float64, device="cuda")
        T.solve(torch.from_numpy(b).cuda(), p, 1e-11, pkg.SolveOpts(precision=prec))
        err = np.linalg.norm((p.cpu().numpy() - p_o)[fl]) / np.linalg.norm(p_o[fl])
        assert err < 1e-8, (prec, err)
    T.close()


@pytest.mark.parametrize("nu1,nu2,inner,krylov", [(2, 2, 2, 0), (1, 0, 1, 0), (1, 2, 3, 0), (0, 2, 2, 0), (2, 1, 1, 8)])
def test_cycles_that_start_from_zero(ctx, nu1, nu2, inner, krylov):
    """A correction cycle's first fused sweep neither reads nor clears e, whichever of the two buffers it is
    in (odd numbers of sweeps swap them) and with values of an earlier solve in both; without a
    pre-smoothing sweep e is cleared.  Against the FP64 solve, on 49 x 37 x 34 cells with a body."""
    pkg, c = ctx
    f = [synth.faces_tanh(m, 1.4) for m in (49, 37, 34)]
    g, T, _, ib, G = classify_both(pkg, c, *f, [synth.ellipsoid(3, (0.2, 0.16, 0.22), 25.0, (0.5, 0.48, 0.51))])
    fl = ib == 0
    for seed in (3, 4):
        b = torch.from_numpy(synth.rhs_divergence(*f, seed)).cuda()
        want = torch.zeros_like(b)
        T.solve(b, want, 1e-11, pkg.SolveOpts(precision=0))
        for prec in (1, 2):
            p = torch.zeros_like(b)
            T.solve(b, p, 1e-11, pkg.SolveOpts(precision=prec, nu1=nu1, nu2=nu2, inner_cycles=inner, krylov=krylov,
                                                    max_cycles=200))
            d = (p - want).cpu().numpy()[fl]
            assert np.linalg.norm(d) < 1e-8 * np.linalg.norm(want.cpu().numpy()[fl]), (seed, prec)
    T.close()


@pytest.mark.parametrize("shape", [(1030, 5, 6), (3, 31, 40), (257, 7, 9), (6, 5, 4)])
def test_packs_by_row_length(ctx, shape):
    """Packs and unpacks take blocks of 1024 consecutive cells: rows longer than a block, many rows in
    a block, a last block in part.  A warm start is met at once and must come back
    as it was but for its mean."""
    pkg, c = ctx
    n = max(shape)
    f = [m / n * synth.faces_tanh(m, 1.2) for m in shape]
    T = pkg.Tables(c, *f, [])
    b = torch.from_numpy(synth.rhs_divergence(*f, 3)).cuda()
    guess = synth.smooth_field(*f, 5) + synth.counter_normal(3, 1, np.arange(b.numel())).reshape(b.shape)
    for prec in (0, 1, 2):
        p = torch.from_numpy(guess.copy()).cuda()
        T.solve(b, p, 1e30, pkg.SolveOpts(precision=prec))   # no cycle: pack, mean, unpack
        d = p.cpu().numpy() - guess                          # minus the mean, a constant
        # pairs carry 48 bits and the difference is rounded a few times
        assert np.max(d) - np.min(d) <= 16 * 2.0**-48 * np.max(np.abs(guess)), prec
    T.close()


@pytest.mark.parametrize("n,r", [(20, 0.11), (56, 0.3), (88, 0.34), (96, 0.36)])
def test_ghost_tables_by_number(ctx, n, r):
    """Eight lanes per ghost up to 8192 ghosts, one above: bit for bit the oracle's tables on both sides."""
    pkg, c = ctx
    f = synth.faces_tanh(n, 1.3)
    _, T, ex, ib, G = classify_both(pkg, c, f, f, f, [synth.octa_sphere(4, (0.5, 0.49, 0.51), r)])
    assert_tables_equal(ex, ib, G)
    T.close()
