"""Box moments against sums over each box's particles, at the sizes around a block's 32
and 256 positions and where the blocks change, read before a walk (which makes the moments
of an FP64 tree) and after it, and the walk after either."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,leaf_cap,sizes", [
    (1, 8, None), (31, 1, None), (32, 8, None), (33, 8, None), (257, 2, None),
    (2500, 40, None), (16384, 8, None), (16385, 8, None), (65536, 16, None),
    (65537, 16, None), (3000, 8, [1, 2000, 999])])
def test_moments(prec, n, leaf_cap, sizes):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(n + (n & 1), 1.0, 3 + n)
    pos, vel, sp = c.pos[:n].copy(), c.vel[:n].copy(), c.species[:n].copy()
    out = []
    for first in (True, False):
        with P.Context(n, c.q, c.m, leaf_cap=leaf_cap, precision=prec, sizes=sizes) as ctx:
            ctx.set_state(pos, vel, sp)
            if first:
                ctx.tree_build()
                g = ctx.get_tree()
            f = ctx.tree_force(0.5, 0.05)
            out.append((ctx.get_tree(), f))
            ids = ctx.get_sorted()[1]
    for k in g:
        assert np.array_equal(g[k], out[0][0][k]) and np.array_equal(g[k], out[1][0][k]), k
    assert all(np.array_equal(a, b) for a, b in zip(out[0][1], out[1][1]))

    x, q = pos[ids], np.array(c.q)[sp[ids]]
    # sums in FP64, or of at most 21 levels' and a leaf's FP32 roundings
    tol = 1e-12 if prec == 0 else 4e-5
    for d in np.unique(g["depth"]):
        i = np.flatnonzero(g["depth"] == d)
        i = i[np.argsort(g["begin"][i])]
        edges = np.stack([g["begin"][i], g["end"][i]], 1).ravel().astype(np.int64)
        box = np.repeat(i, (g["end"] - g["begin"])[i])
        part = np.concatenate([np.arange(b, e) for b, e in edges.reshape(-1, 2)])
        start = np.concatenate([[0], np.cumsum((g["end"] - g["begin"])[i])[:-1]]).astype(np.int64)

        def total(v):
            return np.add.reduceat(v, start, axis=0)

        y, qp = x[part] - g["centre"][box], q[part]
        S0, M = total(np.abs(qp)), total(qp)
        # a box's own scale; FP64 keeps positions to 1e-16 of the cloud's
        s = g["side"][i] if prec else np.full(len(i), g["side"].max())
        e = total(np.abs(qp)[:, None] * y) / S0[:, None]
        assert (np.abs(g["S0"][i] - S0) <= tol * S0).all() and (np.abs(g["M"][i] - M) <= tol * S0).all()
        assert (np.abs(g["c"][i] - g["centre"][i] - e) <= tol * s[:, None]).all()
        assert (np.abs(g["delta"][i] - np.sqrt((e * e).sum(1))) <= 2 * tol * s).all()
        r = x[part] - g["c"][box]
        D = total(qp[:, None] * r)
        Q = total(qp[:, None] * r[:, [0, 0, 0, 1, 1, 2]] * r[:, [0, 1, 2, 1, 2, 2]])
        assert (np.abs(g["D"][i] - D) <= tol * (S0 * s)[:, None]).all()
        assert (np.abs(g["Q"][i] - Q) <= tol * (S0 * s * s)[:, None]).all()
