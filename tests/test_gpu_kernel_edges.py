"""Kernels at the sizes where their work split changes: remainders, tile edges, the smallest and
largest of a range, against the oracle or a plain NumPy statement of the same arithmetic."""
import numpy as np
import pytest

import synth
from oracle import classify as OC
from oracle import forces as OF
from oracle.grid import Grid
from tests.gpu_util import require_gpu, torch

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
