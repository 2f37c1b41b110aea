"""Both forms of the red-black sweep, the fused z-march and the strips, each where it runs.

The two forms leave the same bits, so which one a solve or a batch takes shows only in the number of kernels
it launches; these tests count them, so that a changed threshold cannot leave a form without its test."""
import numpy as np
import pytest

import synth
from tests.gpu_util import require_gpu, torch

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
