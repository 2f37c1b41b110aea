"""Calls over the whole range of sizes they take: results against the oracle at the sizes where the
division of the work changes, and times where a division once suited only some sizes."""
import time

import numpy as np
import pytest

import synth
from oracle import forces as OF
from oracle import system as OY
from tests.gpu_util import classify_both, require_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    require_gpu()
    import paper_2605_04335_gb300 as pkg
    c = pkg.Context(0)
    yield pkg, c
    c.close()


def _best(call, n=7):
    """Shortest of n calls, each waited for, in seconds."""
    t = []
    for _ in range(n + 1):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        call()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t[1:])


@pytest.mark.parametrize("shape", [(2, 33, 18), (3, 9, 20), (4, 17, 33), (5, 8, 5), (8, 31, 17), (9, 30, 40), (12, 40, 33),
                                   (16, 15, 16), (17, 9, 33), (24, 26, 35), (32, 12, 18), (33, 10, 9)])
def test_noalloc_residual_on_short_rows(ctx, shape):
    """Rows of up to 32 cells share a warp (2 to 32 lanes each, the last group of rows in part): against
    the oracle's residual, with a large mean in the right-hand side and p undefined inside the body."""
    pkg, c = ctx
    f = [synth.faces_tanh(m, 1.7) for m in shape]
    meshes = [synth.octa_sphere(2, (0.5, 0.5, 0.5), 0.3)] if min(shape) > 8 else []
    g, T, _, ib, G = classify_both(pkg, c, *f, meshes)
    e = T.export()
    b = synth.counter_normal(3, 0, np.arange(ib.size)).reshape(ib.shape) + 5.0
    p = synth.smooth_field(*f, 4) + 1e-3 * synth.counter_normal(3, 1, np.arange(ib.size)).reshape(ib.shape)
    rel, sr, sb = pkg.ibm_residual_norm_noalloc(*f, e["iblank"], e["cell"], e["ref"], e["w"], e["scale"],
                                                torch.from_numpy(b).cuda(),
                                                torch.from_numpy(np.where(ib == 1, np.nan, p)).cuda())
    rf, rg = OY.residual(g, ib, G, b, p, 0.0)
    want = OY.projected_norm(g, ib, G, rf, rg)
    base = OY.projected_norm(g, ib, G, np.where(ib == 0, b, 0.0), np.zeros(len(G)))
    # a residual cell carries about 10 roundings of sum |c| |p| and of the mean of b
    assert abs(sr - want) <= 1e-12 * want and abs(sb - base) <= 1e-12 * base and abs(rel - want / base) <= 2e-12 * rel
    T.close()


def test_noalloc_residual_takes_short_rows_as_fast_as_long_ones(ctx):
    """The same 4,194,304 cells in rows of 4 and of 1024: no more than twice the time (one row per warp
    took four times as long on the short ones)."""
    pkg, c = ctx
    times = []
    for shape in ((4, 1024, 1024), (1024, 1024, 4)):
        f = [synth.faces_uniform(m) for m in shape]
        T = pkg.Tables(c, *f, [])
        e = T.export()
        b = torch.ones(T.shape, dtype=torch.float64, device="cuda")
        p = torch.arange(b.numel(), dtype=torch.float64, device="cuda").reshape(b.shape) / b.numel()
        times.append(_best(lambda: pkg.ibm_residual_norm_noalloc(*f, e["iblank"], e["cell"], e["ref"], e["w"], e["scale"],
                                                                 b, p)))
        T.close()
    assert times[0] <= 2.0 * times[1], times


def _cone(n, centre, size):
    """Closed double cone of 2 n triangles: two apexes of n triangles each, ring nodes of four."""
    a = 2.0 * np.pi * np.arange(n) / n
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), np.zeros(n)], 1), [[0.0, 0.0, 1.1], [0.0, 0.0, -0.9]]])
    i, j = np.arange(n), (np.arange(n) + 1) % n
    t = np.concatenate([np.stack([i, j, np.full(n, n)], 1), np.stack([j, i, np.full(n, n + 1)], 1)])
    return synth.Mesh(size * v + np.asarray(centre), t[np.random.RandomState(n).permutation(2 * n)].astype(np.int32), 1)


@pytest.mark.parametrize("valences", [(7, 8, 9, 10, 11, 12), (3, 40, 8, 33, 9, 150), (15, 16, 17, 18, 31, 64), (17,) * 6])
def test_nodal_forces_by_triangles_per_node(ctx, valences):
    """One thread per node of up to 16 triangles, a warp per node above (several such nodes in one block):
    bit for bit the oracle's ordered sums."""
    pkg, c = ctx
    f = synth.faces_uniform(30)
    at = [(x, y, z) for z in (0.25, 0.75) for y in (0.3, 0.7) for x in (0.25, 0.75)]
    meshes = [_cone(n, at[q], 0.16 + 0.005 * q) for q, n in enumerate(valences)]
    g, T, _, ib, _ = classify_both(pkg, c, f, f, f, meshes, oracle_ghosts=False)
    p = synth.counter_normal(5, 0, np.arange(ib.size)).reshape(ib.shape)
    out = T.surface_forces(meshes, torch.from_numpy(p).cuda())
    ps, _, F = OF.surface_forces(g, ib, meshes, p)
    assert np.array_equal(out["p_side"].cpu().numpy(), ps)
    assert np.array_equal(out["f_node"].cpu().numpy(), F)
    T.close()



def test_nodal_sums_are_a_small_part_of_a_large_mesh(ctx):
    """262,146 nodes of four or six triangles each: the ordered sums take less of the device than the surface
    pressures of the 524,288 triangles (a warp per node took as long; one thread per node 14 us of 301)."""
    from torch.profiler import ProfilerActivity, profile
    pkg, c = ctx
    f = synth.faces_uniform(64)
    meshes = [synth.octa_sphere(8, (0.5, 0.5, 0.5), 0.33)]
    T = pkg.Tables(c, f, f, f, meshes)
    p = torch.ones(T.shape, dtype=torch.float64, device="cuda")
    for _ in range(2):   # the first profile starts the profiler
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            for _ in range(3):
                T.surface_forces(meshes, p)
            torch.cuda.synchronize()
    t = {k: sum(e.self_device_time_total for e in prof.key_averages() if k in e.key)
         for k in ("k_node_forces", "k_tri_pressure")}
    T.close()
    if not all(t.values()):
        pytest.skip("no kernel times from the profiler")
    assert t["k_node_forces"] <= 0.25 * t["k_tri_pressure"], t
