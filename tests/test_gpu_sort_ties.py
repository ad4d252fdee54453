"""Equal keys in any number come out by caller index: one particle of a stepped cloud leaves
for so far away that every other, by then in the slot order of an earlier tree, shares one
key (in an ensemble: in one of the clouds)."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[3000], [6145], [40000], [500, 9000, 1200]])
def test_one_key_in_slot_order(orc, sizes):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    clouds = [gaussian_cloud(m + m % 2, 1.0, 90 + m) for m in sizes]
    pos, vel, sp = (np.concatenate([getattr(c, a)[:m] for c, m in zip(clouds, sizes)])
                    for a in ("pos", "vel", "species"))
    vel[sizes[0] + 7 if len(sizes) > 1 else 7] = [3e13, -1e13, 2e13]
    n = len(pos)
    with P.Context(n, (1.0, -1.0), (1000.0, 1.0), leaf_cap=32, precision=1,
                   sizes=sizes if len(sizes) > 1 else None) as ctx:
        ctx.set_state(pos, vel, sp)
        ctx.step(1e-3, 1, 1, 0.5, 0.05)
        x, _ = ctx.get_state()
        ctx.tree_build()
        keys, ids = ctx.get_sorted()
    off = 0
    longest = 0
    for m in sizes:
        ok = orc.keys(x[off:off + m], orc.root_cube(x[off:off + m]))
        order = orc.sort_order(ok)
        assert np.array_equal(ids[off:off + m].astype(np.int64) - off, order)
        assert np.array_equal(keys[off:off + m], ok[order])
        longest = max(longest, np.unique(ok, return_counts=True)[1].max())
        off += m
    # (the far corner of the cube cuts cells anywhere: the cloud may lie in a few)
    assert longest >= min(n, 9000) // 8


@pytest.mark.parametrize("n,sizes", [
    (304 * 2048, None), (304 * 2048 + 1, None),       # a tile to every resident block, and one more
    (1300001, None),                                  # four passes over the top digits
    (660000, [640000, 20000])])                       # a ninth pass, by cloud
def test_whole_keys_over_many_tiles(orc, n, sizes):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    pos = np.random.default_rng(n).standard_normal((n, 3))
    pos[n // 3] = [1e3, 2e4, -3e3]
    sp = (np.arange(n) % 2).astype(np.int8)
    with P.Context(n, (1.0, -1.0), (1000.0, 1.0), leaf_cap=32, precision=1, sizes=sizes) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        ctx.tree_build()
        keys, ids = ctx.get_sorted()
        x, _ = ctx.get_state()
    assert np.array_equal(x, pos)
    off = 0
    for m in sizes or [n]:
        ok = orc.keys(pos[off:off + m], orc.root_cube(pos[off:off + m]))
        order = orc.sort_order(ok)
        assert np.array_equal(ids[off:off + m].astype(np.int64) - off, order)
        assert np.array_equal(keys[off:off + m], ok[order])
        off += m
