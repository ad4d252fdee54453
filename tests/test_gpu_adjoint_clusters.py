"""FP32C vector-Jacobian products of small clusters far apart, where groups of targets lie over
the gaps: within the rounding of the FP32 form (ten powers of a distance known to 2^-24: under
1e-6 rms) of the FP64 context's, as in a single cloud."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,clusters,leaf_cap,theta", [
    (2500, 200, 1, 0.5), (2500, 200, 1, 0.9), (1001, 90, 4, 0.5), (20001, 600, 16, 0.6)])
def test_clusters(n, clusters, leaf_cap, theta):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    rng = np.random.default_rng(n)
    pos = 0.01 * rng.standard_normal((n, 3)) + \
        50.0 * rng.standard_normal((clusters, 3))[np.arange(n) % clusters]
    sp = (np.arange(n) % 2).astype(np.int8)
    lam = rng.standard_normal((n, 3))
    mu = []
    for prec in (0, 1):
        with P.Context(n, (1.0, -1.0), (10.0, 1.0), leaf_cap=leaf_cap, precision=prec) as ctx:
            ctx.set_state(pos, np.zeros_like(pos), sp)
            mu.append(ctx.accel_vjp(theta, 0.05, lam))
    assert np.sqrt(((mu[1] - mu[0]) ** 2).sum() / (mu[0] ** 2).sum()) <= 1e-6
