"""FP64 contexts decide Eq. 5 as FP64 does in every unit of length: a cloud, its softening
and its expansion scaled by a power of two (all exact) open and accept the same boxes, also
where squares leave the range of FP32, and forces and their derivatives scale with it."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


def _walk(P, c, f, theta, leaf_cap, with_vjp):
    with P.Context(c.n, c.q, c.m, leaf_cap=leaf_cap, precision=0) as ctx:
        ctx.set_state(c.pos * f, c.vel, c.species)
        acc, phi = ctx.tree_force(theta, 0.01 * f)
        counts = ctx.get_counts()
        mu = ctx.accel_vjp(theta, 0.01 * f, np.cos(c.vel)) if with_vjp else np.zeros(1)
    return acc, phi, counts, mu


@pytest.mark.parametrize("theta,leaf_cap", [(0.5, 8), (1.0, 1), (0.0, 4)])
@pytest.mark.parametrize("scale", [-80, -40, -10, 22, 40, 63, 64, 70, 127, 140])
def test_scaled_cloud(theta, leaf_cap, scale):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(1000, 1.0, 77)
    # (at scales past 2^70 the derivative's ninth power of 1/r leaves the range of FP64)
    vjp = abs(scale) <= 80
    f = 2.0 ** scale
    acc, phi, counts, mu = _walk(P, c, f, theta, leaf_cap, vjp)
    ref, ref_phi, ref_counts, ref_mu = _walk(P, c, 1.0, theta, leaf_cap, vjp)
    assert np.array_equal(counts[0], ref_counts[0]) and np.array_equal(counts[1], ref_counts[1])
    # the same operations but for the reciprocal root, an ulp apart: sums of 1e3 terms
    assert np.abs(acc * f * f - ref).max() <= 1e-13 * np.abs(ref).max()
    assert np.abs(phi * f - ref_phi).max() <= 1e-13 * np.abs(ref_phi).max()
    if vjp:
        assert np.abs(mu * f ** 3 - ref_mu).max() <= 1e-12 * np.abs(ref_mu).max()
