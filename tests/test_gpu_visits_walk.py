"""The walk of the gradient's forward runs: one and two warps to a chunk give the same run
bit for bit (the same cloud alone and inside an ensemble of 70,000 more particles), and
that run is the ordinary push's to the rounding of its FP32 sums."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf_cap,theta,fat", [
    (2, 1, 0.5, 0), (33, 1, 1.0, 0), (700, 1, 0.0, 0), (4099, 16, 0.5, 0),
    (3001, 300, 0.6, 0),        # leaves longer than the shared buffer
    (2000, 4, 0.4, 333),        # a leaf of coincident particles
    (19456, 32, 0.5, 0), (38000, 2, 0.8, 0)])
def test_visits_walk(n, leaf_cap, theta, fat):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c, d = gaussian_cloud(n + (n & 1), 1.0, 5 + n), gaussian_cloud(70000, 2.0, 6)
    pos, vel, sp = c.pos[:n].copy(), c.vel[:n].copy(), c.species[:n].copy()
    if fat:
        pos[:fat] = pos[0]
    dt, k, eps = 1e-4, 2, 0.05
    out = []
    for sizes in (None, [n, 70000]):
        state = [pos, vel, sp] if sizes is None else \
            [np.concatenate(v) for v in ((pos, d.pos), (vel, d.vel), (sp, d.species))]
        with P.Context(len(state[0]), c.q, c.m, leaf_cap=leaf_cap, precision=1, sizes=sizes) as ctx:
            ctx.set_state(*state)
            ctx.grad_ke_electrons(dt, k, 2 * k, theta, eps, k)
            out.append([v[:n] for v in ctx.get_state()])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    with P.Context(n, c.q, c.m, leaf_cap=leaf_cap, precision=1) as ctx:
        ctx.set_state(pos, vel, sp)
        a0, _ = ctx.tree_force(theta, eps)
        ctx.step(dt, k, 2 * k, theta, eps)
        p, v = ctx.get_state()
    # both sums are within 1e-6 of the largest acceleration of each other
    a = np.abs(a0).max()
    assert np.abs(out[0][1] - v).max() <= 1e-6 * a * 2 * k * dt
    assert np.abs(out[0][0] - p).max() <= 1e-6 * a * (2 * k * dt) ** 2 + 1e-15 * np.abs(pos).max()
