"""Both forms of the red-black sweep, the fused z-march and the strips, each where it runs.

The two forms leave the same bits, so which one a solve or a batch takes shows only in the number of kernels
it launches; these tests count them, so that a changed threshold cannot leave a form without its test."""
import numpy as np
import pytest

import synth
from tests.gpu_util import require_gpu, torch
from tests.test_gpu_sweep import _check

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    import paper_2605_04335_gb300 as pkg
    c = pkg.Context(0)
    yield pkg, c
    c.close()


def _problem(pkg, c, shape, seed, body=0.3):
    """Cubic cells, a sphere; its tables and right-hand side."""
    n = max(shape)
    f = [np.arange(m + 1) / n for m in shape]
    mid = [0.5 * m / n + 0.003 * ((seed + a) % 5) for a, m in enumerate(shape)]
    T = pkg.Tables(c, *f, [synth.octa_sphere(3, mid, body * min(shape) / n)])
    return T, torch.from_numpy(synth.rhs_divergence(*f, seed)).cuda()


def _batch_launches(pkg, c, tabs, rhs, steps, **o):
    """Kernels of a lockstep batch held to so many steps."""
    n0 = pkg.ibm_ctx_launch_count(c.h)
    status, reps = pkg.poisson_solve_batched(c.h, [t.h for t in tabs], rhs, 1e-15, [torch.zeros_like(b) for b in rhs],
                                             pkg.SolveOpts(precision=1, max_cycles=steps, **o), raise_on_error=False)
    assert all(r["cycles"] == steps for r in reps), (status, reps)
    return pkg.ibm_ctx_launch_count(c.h) - n0


def _launches_per_step(pkg, c, tabs, rhs, **o):
    _batch_launches(pkg, c, tabs, rhs, 1, **o)   # hierarchies
    return _batch_launches(pkg, c, tabs, rhs, 3, **o) - _batch_launches(pkg, c, tabs, rhs, 2, **o)


def _close(tabs):
    for t in tabs:
        t.close()


def test_batch_of_two_sizes_takes_one_form(ctx):
    """Problems of 30^3 and 34^3 cells, either side of 2^15, share each stage's launch: the mixed batch launches per
    step what two problems of 34^3 launch, and the coarse tail of the smaller one (from one level earlier) once per
    V-cycle.  Each problem gets its own solve's bits."""
    pkg, c = ctx
    a, b = (_problem(pkg, c, (n, n, n), n) for n in (30, 34))
    d = _problem(pkg, c, (34, 34, 34), 35)
    tabs, rhs = zip(a, b)
    assert _launches_per_step(pkg, c, tabs, rhs) == _launches_per_step(pkg, c, (b[0], d[0]), (b[1], d[1])) + 2
    ps = [torch.zeros_like(r) for r in rhs]
    pkg.poisson_solve_batched(c.h, [t.h for t in tabs], rhs, TOL, ps, pkg.SolveOpts(precision=1))
    for t, r, p in zip(tabs, rhs, ps):
        own = torch.zeros_like(r)
        t.solve(r, own, TOL, pkg.SolveOpts(precision=1))
        assert torch.equal(own, p)
    _close([a[0], b[0], d[0]])


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("nu1,nu2,inner", [(2, 1, 1), (1, 0, 1), (2, 2, 2)])
def test_small_solves_of_odd_schedules(ctx, prec, nu1, nu2, inner):
    """Steps of an odd number of sweeps on at most 2^15 cells are relaxed by strips and replayed as a graph: the same
    bits as launched directly, and as the fused sweep leaves them in a batch of the one problem."""
    pkg, c = ctx
    T, b = _problem(pkg, c, (26, 31, 22), 3)
    out = []
    for graph in (1, 0):
        p = torch.zeros_like(b)
        T.solve(b, p, TOL, pkg.SolveOpts(precision=prec, nu1=nu1, nu2=nu2, inner_cycles=inner, use_graph=graph, max_cycles=200))
        out.append(p)
    p = torch.zeros_like(b)
    pkg.poisson_solve_batched(c.h, [T.h], [b], TOL, [p],
                              pkg.SolveOpts(precision=prec, nu1=nu1, nu2=nu2, inner_cycles=inner, max_cycles=200))
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], p)
    T.close()


def _sphere_at(xf, yf, zf, i, j, k, r):
    return synth.octa_sphere(4, (xf[i], yf[j], 0.5 * (zf[k] + zf[k + 1])), r)


@pytest.mark.parametrize("shape,prec,fused", [((200, 83, 65), 0, True), ((128, 96, 85), 0, False), ((200, 45, 37), 1, True),
                                              ((37, 20, 9), 1, True), ((37, 20, 9), 2, True), ((5, 4, 6), 1, True)])
def test_form_of_the_finest_sweep(ctx, shape, prec, fused):
    """Fused: one kernel per sweep and one for the ghost rows; strips: one per colour, and two for the ghost rows.
    FP64 fused from 2^20 cells, FP32 whatever the size."""
    pkg, c = ctx
    T, b = _problem(pkg, c, shape, 3)
    n = []
    for sweeps in (1, 1, 2):   # the first builds the hierarchy
        n0 = pkg.ibm_ctx_launch_count(c.h)
        pkg.ibm_smoother_apply(c.h, T.h, prec, sweeps, 1.3, torch.zeros_like(b), b, 0.0)
        n.append(pkg.ibm_ctx_launch_count(c.h) - n0)
    ghosts = T.nghost > 0
    assert n[2] - n[1] == (1 + ghosts if fused else 2 + 2 * ghosts), (n, T.nghost)
    T.close()


def test_fused_fp64_sweep_across_tile_borders(ctx):
    """200 x 83 x 65 cells in FP64 (the fused form, as its launches show above): 2 x 6 tiles, both ragged, bodies over the
    x = 128 and y = 14, 42 borders and over chunk seams in z."""
    xf, yf, zf = synth.faces_tanh(200, 1.5), synth.faces_uniform(83), synth.faces_tanh(65, 1.2)
    _check(ctx, xf, yf, zf, [_sphere_at(xf, yf, zf, 128, 42, 31, 0.17), _sphere_at(xf, yf, zf, 60, 14, 20, 0.08)], 41,
           precisions=(0,))


def test_fused_fp64_sweep_without_a_body(ctx):
    """301 x 57 x 62 cells in FP64, no body: three tiles in x and five in y, the last of each ragged."""
    _check(ctx, synth.faces_uniform(301), synth.faces_tanh(57, 2.0), synth.faces_tanh(62, 1.4), [], 42, precisions=(0,))


@pytest.fixture
def coarse_line(ctx):
    """Sets the cells from which coarse levels take the fused sweep; the normal line afterwards."""
    pkg, c = ctx
    yield lambda cells: pkg.ibm_ctx_set_coarse_fused_cells(c.h, cells)
    pkg.ibm_ctx_set_coarse_fused_cells(c.h, -1)


def _solve_both(pkg, c, coarse_line, shape, seed, prec):
    """(p, report, kernels launched) by strips and by the fused sweep on level 1."""
    out = []
    for line in (-1, 1 << 18):
        coarse_line(line)
        T, b = _problem(pkg, c, shape, seed, 0.36)
        for _ in range(2):   # the first builds the hierarchy
            p = torch.zeros_like(b)
            n0 = pkg.ibm_ctx_launch_count(c.h)
            rep = T.solve(b, p, TOL, pkg.SolveOpts(precision=prec, use_graph=0))
            n = pkg.ibm_ctx_launch_count(c.h) - n0
        out.append((p, rep, n))
        T.close()
    return out


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("shape", [(300, 64, 130), (140, 132, 126)])
def test_fused_coarse_level_leaves_the_bits_of_the_strips(ctx, coarse_line, shape, prec):
    """Level 1 of 150 x 32 x 65 (two by three tiles, a body over their borders) and of 70 x 66 x 63 cells: the solve's
    pressure, cycles and history are the strips' bit for bit, with one kernel less for each of the eight sweeps
    a step takes on the level."""
    pkg, c = ctx
    (p0, r0, n0), (p1, r1, n1) = _solve_both(pkg, c, coarse_line, shape, 5, prec)
    assert r0["cycles"] == r1["cycles"] and np.array_equal(r0["history"], r1["history"])
    assert torch.equal(p0, p1)
    assert n0 - n1 == 8 * r0["cycles"], (n0, n1, r0["cycles"])


def test_fused_coarse_level_in_lockstep(ctx, coarse_line):
    """The batched form of the coarse fused sweep, two problems of other shapes in one launch: each problem's pressure is
    its own solve's, by strips, bit for bit."""
    pkg, c = ctx
    shapes = [(300, 64, 130), (140, 132, 126)]
    coarse_line(-1)
    want = []
    for q, shape in enumerate(shapes):
        T, b = _problem(pkg, c, shape, q, 0.36)
        p = torch.zeros_like(b)
        want.append((p, T.solve(b, p, TOL, pkg.SolveOpts(precision=1))))
        T.close()
    steps = []
    for line in (-1, 1 << 18):
        coarse_line(line)
        tabs, rhs = zip(*(_problem(pkg, c, shape, q, 0.36) for q, shape in enumerate(shapes)))
        ps = [torch.zeros_like(b) for b in rhs]
        _, reps = pkg.poisson_solve_batched(c.h, [t.h for t in tabs], rhs, TOL, ps, pkg.SolveOpts(precision=1))
        for p, rep, (w, r) in zip(ps, reps, want):
            assert rep["cycles"] == r["cycles"] and torch.equal(p, w)
        steps.append(_launches_per_step(pkg, c, tabs, rhs))
        _close(tabs)
    assert steps[0] - steps[1] == 8, steps


@pytest.mark.parametrize("count,shapes,by_strips", [(12, [(96, 88, 90), (90, 97, 85)], False), (38, [(32, 31, 31), (31, 32, 29)], True)])
def test_lockstep_strips_of_two_planes(ctx, count, shapes, by_strips):
    """Strips take two planes per thread where a launch holds 2^20 cells or more, here by the sum over the batch (level 1
    of 12 problems; the finest level of 38) of levels that take one plane in their own solves, with odd numbers of
    planes: every problem gets its own solve's bits."""
    pkg, c = ctx
    level = [tuple((n + (not by_strips)) // (1 if by_strips else 2) for n in shapes[q % 2]) for q in range(count)]
    assert sum(int(np.prod(s)) for s in level) >= 1 << 20 and all(np.prod(s) < 1 << 18 for s in level)
    assert any(s[2] % 2 for s in level)
    tabs, rhs = zip(*(_problem(pkg, c, shapes[q % 2], q) for q in range(count)))
    few = _launches_per_step(pkg, c, tabs[:2], rhs[:2])
    # strips: two kernels more per sweep of the finest level (its ghost rows too), and one that clears e
    assert _launches_per_step(pkg, c, tabs, rhs) - few == (8 * 2 + 1 if by_strips else 0)
    ps = [torch.zeros_like(b) for b in rhs]
    _, reps = pkg.poisson_solve_batched(c.h, [t.h for t in tabs], rhs, TOL, ps, pkg.SolveOpts(precision=1))
    for t, b, p, rep in zip(tabs, rhs, ps, reps):
        own = torch.zeros_like(b)
        r = t.solve(b, own, TOL, pkg.SolveOpts(precision=1))
        assert r["cycles"] == rep["cycles"] and torch.equal(own, p)
    _close(tabs)
