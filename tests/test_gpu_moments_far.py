"""FP64 centroids and dipoles where the boxes are small against the cube and its distance from
the origin is not theirs: a dense core, a particle far out, a core away from the cube's centre.
Exact values by extended-precision sums over each box's particles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cloud(name):
    rng = np.random.default_rng(17)
    x = rng.standard_normal((1500, 3))
    if name == "core":
        return x ** 5
    if name == "far":
        x[3] = [2e5, -3e4, 1e5]
        return x
    x[:700] = 300.0 + 1e-3 * x[:700]
    return x


@pytest.mark.parametrize("name", ["core", "far", "two"])
@pytest.mark.parametrize("leaf_cap", [1, 8])
def test_centroids(name, leaf_cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    pos = _cloud(name)
    n = len(pos)
    q, m = (1.5, -0.7), (10.0, 1.0)
    sp = (np.arange(n) % 3 == 0).astype(np.int8)
    with P.Context(n, q, m, leaf_cap=leaf_cap, precision=0) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        ctx.tree_build()
        tree = ctx.get_tree()
        _, ids = ctx.get_sorted()
    x = pos[ids].astype(np.longdouble)
    qs = np.asarray(q, dtype=np.longdouble)[sp[ids]]
    eps = 2.0 ** -53
    for i, (b, e) in enumerate(zip(tree["begin"], tree["end"])):
        w = np.abs(qs[b:e])
        c = (w[:, None] * x[b:e]).sum(0) / w.sum()
        # offsets of at most a side, rounded and summed over levels and children (under 60
        # roundings of side / 2), and the centroid's own rounding
        off = np.abs(tree["c"][i] - c).max()
        tol = eps * (30.0 * tree["side"][i] + 2.0 * float(np.abs(c).max()))
        assert off <= tol, (i, float(off / tol))
        # the dipole about c: the same offsets and their errors, times the charges
        d = (qs[b:e][:, None] * (x[b:e] - c)).sum(0)
        assert np.abs(tree["D"][i] - d).max() <= eps * float(w.sum()) * 60.0 * tree["side"][i]
