"""The key order of small clouds, sorted by one block, at its sizes' edges and beyond its
largest: runs of equal top digits up to, at and past the length that is ordered in place,
coincident particles (ties by caller index, also after a step has reordered the slots).
Keys, order and cube are the oracle's, bit for bit."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


def _positions(n, kind):
    rng = np.random.default_rng(n)
    pos = gaussian_cloud(n + (n & 1), 1.0, 9).pos[:n].copy()
    if kind == "coincident":
        pos[n // 3:] = pos[rng.integers(0, 1 + n // 40, n - n // 3)]
    elif kind == "one place":
        pos[:] = pos[0]
    elif kind != "cloud":                       # tight groups of `kind`, in random order
        pos = np.repeat(rng.uniform(-1, 1, (n // kind + 1, 3)), kind, axis=0)[:n]
        pos = rng.permutation(pos + 1e-9 * rng.uniform(-1, 1, pos.shape))
    return np.ascontiguousarray(pos)


@pytest.mark.parametrize("kind", ["cloud", "coincident", "one place", 32, 33])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1025, 4097, 6143, 6144, 6145, 8192, 10007])
def test_block_sort(orc, n, kind):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    pos = _positions(n, kind)
    sp = (np.arange(n) % 2).astype(np.int8)
    vel = np.random.default_rng(1).standard_normal((n, 3))
    with P.Context(n, (1.0, -1.0), (1000.0, 1.0), leaf_cap=32, precision=1) as ctx:
        ctx.set_state(pos, vel, sp)
        for first in (True, False):
            ctx.tree_build()
            keys, ids = ctx.get_sorted()
            p, v = ctx.get_state()
            ok = orc.keys(p, orc.root_cube(p))
            order = orc.sort_order(ok)
            assert np.array_equal(ids.astype(np.int64), order)
            assert np.array_equal(keys, ok[order])
            if first:
                assert np.array_equal(p, pos) and np.array_equal(v, vel)
            ctx.step(1e-4, 1, 1, 1.0, 0.5)
