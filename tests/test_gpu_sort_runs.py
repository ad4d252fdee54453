"""The key sort's runs of equal top digits: runs at and beyond the length that is ordered
in shared memory (32), across the blocks' places, over whole clouds (one far particle puts
every other into one cell), ensembles, every number of passes, and replays as captured
graphs.  Keys and order are the oracle's, bit for bit."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def U():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0709_3331_gb300 import build as b
    b.build()
    import paper_0709_3331_gb300 as P
    return P


def _clusters(sizes, n, seed):
    """Tight groups (within 1e-9 of a random place) of the given sizes, in random order."""
    rng = np.random.default_rng(seed)
    pos = []
    while sum(len(p) for p in pos) < n:
        m = sizes[len(pos) % len(sizes)]
        pos.append(rng.uniform(-1, 1, 3) + 1e-9 * rng.uniform(-1, 1, (m, 3)))
    return rng.permutation(np.concatenate(pos)[:n])


def _case(name):
    if name == "outlier":
        pos = gaussian_cloud(20000, 1.0, 5).pos
        pos[777] = [3e6, -1e6, 2e6]
    elif name == "outlier_small":
        pos = gaussian_cloud(600, 1.0, 6).pos
        pos[0] = 1e9
    elif name == "runs_of_32":
        pos = _clusters([1, 31, 32, 2, 32, 7], 6007, 1)
    elif name == "runs_of_33":
        pos = _clusters([1, 32, 33, 2], 5003, 2)
    elif name == "runs_of_300":
        pos = _clusters([300, 1, 5], 4500, 3)
    elif name == "coincident":
        pos = gaussian_cloud(3000, 1.0, 7).pos
        pos[10:90] = pos[10]
        pos[1000::100] = pos[1000]
    elif name == "four_passes":
        pos = gaussian_cloud(1100000, 10.0, 8).pos
    elif name == "three_passes_dense":
        pos = gaussian_cloud(1000000, 10.0, 9).pos ** 3     # denser centre: longer runs
    else:
        pos = gaussian_cloud(4, 1.0, 10).pos[:int(name)]
    return np.ascontiguousarray(pos)


@pytest.mark.parametrize("name", ["outlier", "outlier_small", "runs_of_32", "runs_of_33",
                                  "runs_of_300", "coincident", "four_passes",
                                  "three_passes_dense", "1", "2", "3"])
def test_order_is_the_oracles(U, orc, name):
    pos = _case(name)
    n = pos.shape[0]
    vel = np.random.default_rng(0).standard_normal((n, 3))
    sp = (np.arange(n) % 2).astype(np.int8)
    with U.Context(n, (1.0, -1.0), (1000.0, 1.0), leaf_cap=32, precision=1) as ctx:
        ctx.set_state(pos, vel, sp)
        ctx.tree_build()
        keys, ids = ctx.get_sorted()
        p, v = ctx.get_state()
    ok = orc.keys(pos, orc.root_cube(pos))
    order = orc.sort_order(ok)
    assert np.array_equal(ids.astype(np.int64), order)
    assert np.array_equal(keys, ok[order])
    assert np.array_equal(p, pos) and np.array_equal(v, vel)


def test_ensemble_with_a_far_particle(U, orc):
    sizes = [700, 5000, 33, 1200]
    clouds = [gaussian_cloud(n + n % 2, 1.0, 60 + n).pos[:n].copy() for n in sizes]
    clouds[1][17] = 1e7
    pos = np.concatenate(clouds)
    n = len(pos)
    sp = (np.arange(n) % 2).astype(np.int8)
    with U.Context(n, (1.0, -1.0), (1000.0, 1.0), leaf_cap=8, precision=1, sizes=sizes) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        ctx.tree_build()
        keys, ids = ctx.get_sorted()
    off = 0
    for x in clouds:
        ok = orc.keys(x, orc.root_cube(x))
        order = orc.sort_order(ok)
        sl = slice(off, off + len(x))
        assert np.array_equal(ids[sl].astype(np.int64) - off, order)
        assert np.array_equal(keys[sl], ok[order])
        off += len(x)


def test_replayed_blocks_with_a_far_particle(U, orc):
    """The device decides at every replay whether the whole key is sorted."""
    c = gaussian_cloud(6000, 1.0, 71)
    far = c.pos.copy()
    far[123] = [2e6, 0.0, -1e6]
    out = []
    for graphs in (False, True):
        with U.Context(c.n, c.q, c.m, leaf_cap=16, precision=1) as ctx:
            ctx.set_graphs(graphs)
            res = []
            for pos in (c.pos, far, c.pos):
                ctx.set_state(pos, c.vel, c.species)
                ctx.step(1e-3, 3, 9, 0.5, 0.05)
                p, v = ctx.get_state()
                ctx.tree_build()
                _, ids = ctx.get_sorted()
                ok = orc.keys(p, orc.root_cube(p))
                assert np.array_equal(ids.astype(np.int64), orc.sort_order(ok))
                res += [p, v]
            out.append(res)
    for a, b in zip(*out):
        assert np.array_equal(a, b)
