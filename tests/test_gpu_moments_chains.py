"""Moments of trees whose twigs have one or two children nearly everywhere: close pairs and
triples in leaves of 1 (chains of up to 20 boxes), particles on a line.  Every 17th box against
extended-precision sums over its particles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cloud(name, n):
    rng = np.random.default_rng(23)
    x = rng.standard_normal((n, 3))
    if name == "pairs":
        x[1::2] = x[0::2] + 1e-6 * x[1::2]
    elif name == "triples":
        x[1::3] = x[0::3][:len(x[1::3])] + 1e-5 * x[1::3]
        x[2::3] = x[0::3][:len(x[2::3])] + 1e-5 * x[2::3]
    else:
        x[:, 1:] = 0.25
    return x


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [2400, 18000, 70002])      # blocks of 32 and of 256 positions
@pytest.mark.parametrize("name", ["pairs", "triples", "line"])
def test_chains(prec, n, name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    pos = _cloud(name, n)
    q = (1.5, -0.7)
    sp = (np.arange(n) % 2).astype(np.int8)
    with P.Context(n, q, (10.0, 1.0), leaf_cap=1, precision=prec) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        ctx.tree_build()
        tree = ctx.get_tree()
        _, ids = ctx.get_sorted()
    x = pos[ids].astype(np.longdouble)
    qs = np.asarray(q, dtype=np.longdouble)[sp[ids]]
    # roundings: a few per level and child, under 60 of half a side for the first moments,
    # twice that for the second; the FP64 centre itself, and what that does to D, one of |c|
    u = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    for i in range(0, len(tree["begin"]), 17):
        b, e, s = tree["begin"][i], tree["end"][i], tree["side"][i]
        w = np.abs(qs[b:e])
        S0 = float(w.sum())
        assert abs(tree["S0"][i] - S0) <= 30 * u * S0
        assert abs(tree["M"][i] - float(qs[b:e].sum())) <= 30 * u * S0
        c = (w[:, None] * x[b:e]).sum(0) / w.sum()
        off = 2.0 ** -53 * 2.0 * float(np.abs(c).max())
        assert np.abs(tree["c"][i] - c).max() <= 30 * u * s + off
        y = x[b:e] - c
        assert np.abs(tree["D"][i] - (qs[b:e][:, None] * y).sum(0)).max() <= S0 * (60 * u * s + off)
        k = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
        Q = np.array([(qs[b:e] * y[:, f] * y[:, g]).sum() for f, g in k])
        assert np.abs(tree["Q"][i] - Q).max() <= S0 * s * (120 * u * s + 2 * off)
