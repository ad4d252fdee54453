"""The FP32 adjoint walk at every number of targets to a warp, on both sides of each size
where it changes, against the FP64 context's (the same interactions), to the FP32 walk's
tolerance; and with chunks taken in the order a walk has left."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,leaf_cap,theta", [
    (2, 1, 0.5), (33, 4, 0.7), (47, 40, 0.5), (4863, 16, 0.5), (4865, 300, 0.6),
    (20001, 2, 0.9), (48639, 32, 0.7), (48641, 32, 0.7)])
def test_groups_of_targets(n, leaf_cap, theta):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(n + (n & 1), 1.0, 31 + n)
    pos, vel, sp = c.pos[:n].copy(), c.vel[:n].copy(), c.species[:n].copy()
    lam = np.random.default_rng(n).standard_normal((n, 3))
    out = []
    for prec in (0, 1, 1):
        with P.Context(n, c.q, c.m, leaf_cap=leaf_cap, precision=prec) as ctx:
            ctx.set_state(pos, vel, sp)
            if len(out) == 2:
                ctx.tree_force(theta, 0.05)     # leaves its order of chunks
            out.append(ctx.accel_vjp(theta, 0.05, lam))
    for mu in out[1:]:
        assert np.sqrt(((mu - out[0]) ** 2).sum() / (out[0] ** 2).sum()) <= 1e-4
