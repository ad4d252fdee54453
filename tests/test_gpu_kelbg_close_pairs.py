"""Electron-ion pairs of the Kelbg law from far apart to as close as FP32 separations go, in
FP32C contexts: potential (1 - e^-u) / r and field [1 - (1 + u) e^-u] / r^2, u = r / lambda,
which tend to 1 / lambda and 1 / (2 lambda^2).  Pairs as an ensemble of two-particle clouds,
so that each separation is exact to an ulp of its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _law(d, lam):
    u = d / lam
    # u < 1e-2: series to u^3 (next term below 1e-10)
    s = u < 1e-2
    us = np.where(s, u, 1.0)
    phi = np.where(s, 1 - us / 2 + us ** 2 / 6 - us ** 3 / 24, -np.expm1(-u) / u) / lam
    f = np.where(s, 0.5 - us / 3 + us ** 2 / 8 - us ** 3 / 30,
                 (-np.expm1(-u) - u * np.exp(-u)) / u ** 2) / lam ** 2
    return phi, f


@pytest.mark.parametrize("lam,lo", [(1.0, -18.0), (0.05, -18.0), (300.0, -18.0), (1e-11, -15.5)])
def test_pairs(lam, lo):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    m = 256
    d = 10.0 ** np.linspace(lo, np.log10(lam) + 1.5, m)
    pos = np.zeros((2 * m, 3))
    pos[1::2] = d[:, None] * np.array([0.6, 0.0, -0.8])
    sp = np.tile(np.array([0, 1], dtype=np.int8), m)
    with P.Context(2 * m, (1.0, -1.0), (1.0, 1.0), leaf_cap=8, precision=1, sizes=[2] * m,
                   kelbg_lambda=lam) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        acc, phi = ctx.tree_force(0.0, 0.01 * lam)
    want_phi, want_f = _law(d, lam)
    # FP32: rsqrt (2 ulp), exp, the series' and the products' roundings, under 40 x 2^-24;
    # from u = 1/2 on, 1 - (1 + u) e^-u cancels to 0.09 of its terms at worst
    tol = 40 * 2.0 ** -24
    assert (np.abs(-phi[0::2] / want_phi - 1) <= tol).all()
    assert (np.abs(phi[1::2] / want_phi - 1) <= tol).all()
    for k, e in ((0, 0.6), (2, -0.8)):
        assert (np.abs(acc[0::2, k] / (e * want_f) - 1) <= tol).all()
        assert (np.abs(acc[1::2, k] / (-e * want_f) - 1) <= tol).all()


def test_below_the_normal_range():
    """r^2 below the smallest normal float keeps few bits: the limits to 1 % at 1e-21."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    d = np.array([0.0, 1e-21, 1e-20, 1e-19])
    pos = np.zeros((8, 3))
    pos[1::2, 1] = d
    sp = np.tile(np.array([0, 1], dtype=np.int8), 4)
    with P.Context(8, (1.0, -1.0), (1.0, 1.0), leaf_cap=8, precision=1, sizes=[2] * 4,
                   kelbg_lambda=0.5) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        acc, phi = ctx.tree_force(0.0, 0.01)
    assert (np.abs(-phi[0::2] / 2.0 - 1) <= 1e-2).all()
    assert acc[0, 1] == 0.0 and acc[1, 1] == 0.0
    assert (np.abs(acc[2::2, 1] / 2.0 - 1) <= 1e-2).all()
