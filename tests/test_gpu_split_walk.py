"""FP32C walks with several warps to a chunk: at every number of warps, and on both sides
of each size where it changes, the results are those of one warp per chunk bit for bit.
The same cloud inside an ensemble of 60,000 more particles takes that form."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kelbg", [None, 0.05])
@pytest.mark.parametrize("n,leaf_cap,theta,fat", [
    (1, 1, 0.5, 0), (33, 1, 1.0, 0), (700, 1, 0.0, 0),
    (3001, 300, 0.6, 0),        # leaves longer than the shared buffer
    (2000, 4, 0.4, 333),        # a leaf of coincident particles
    (9728, 16, 0.5, 0), (9729, 16, 0.5, 0), (19456, 16, 0.5, 0), (19457, 32, 0.5, 0),
    (24320, 32, 0.5, 0), (24321, 32, 0.5, 0), (48640, 32, 0.5, 0), (48641, 32, 0.5, 0)])
def test_split_walk(kelbg, n, leaf_cap, theta, fat):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c, d = gaussian_cloud(n + (n & 1), 1.0, 5 + n), gaussian_cloud(60000, 2.0, 6)
    pos, vel, sp = c.pos[:n].copy(), c.vel[:n].copy(), c.species[:n].copy()
    if fat:
        pos[:fat] = pos[0]
    out = []
    for sizes in (None, [n, 60000]):
        state = [pos, vel, sp] if sizes is None else \
            [np.concatenate(v) for v in ((pos, d.pos), (vel, d.vel), (sp, d.species))]
        with P.Context(len(state[0]), c.q, c.m, leaf_cap=leaf_cap, precision=1, sizes=sizes,
                       kelbg_lambda=kelbg) as ctx:
            ctx.set_state(*state)
            res = ctx.tree_force(theta, 0.05) + ctx.get_counts()
            ctx.step(1e-4, 2, 2, theta, 0.05)       # the electrons alone, then every particle
            res += ctx.get_state()
        out.append([v[:n] for v in res])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
