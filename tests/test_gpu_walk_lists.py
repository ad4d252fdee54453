"""The walks' lists at their edges, against the oracle: the stack of opened twigs
past its wide limit (small theta, one-particle leaves), leaves longer than one part of
the shared buffer (32 sources), odd sizes and targets fewer than a warp, clouds of
coincident particles.  The tolerances are the walks' own (1e-5 FP64, 1e-4 FP32C, force
relative RMS); the interaction counts are the oracle's except where a decision lies
within the rounding of a pseudo-particle's position (0.1 % + 2 targets)."""
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


def rel_rms(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


@pytest.mark.parametrize("prec,tol", [(0, 1e-5), (1, 1e-4)])
@pytest.mark.parametrize("n,leaf_cap,theta,fat", [
    (4096, 1, 0.0, 0),      # every twig opened: the stack at its largest
    (2999, 1, 0.1, 0),
    (5001, 64, 0.5, 0),     # leaves of 33 to 64 sources
    (3000, 300, 0.6, 0),    # several parts per leaf, shallow tree
    (2000, 4, 0.4, 333),    # a depth-21 leaf of 333 coincident particles
    (31, 1, 0.5, 0),
    (3, 1, 1.0, 0),
])
def test_walk_lists(U, orc, prec, tol, n, leaf_cap, theta, fat):
    c = gaussian_cloud(n + (n & 1), 1.0, 101 + n)
    pos, vel, sp = c.pos[:n].copy(), c.vel[:n].copy(), c.species[:n].copy()
    if fat:
        pos[:fat] = pos[0]
    eps = 0.05
    E, phi, npp, nmp = orc.Tree(pos, sp, c.q, leaf_cap=leaf_cap).force(theta, eps, counts=True,
                                                                       nthreads=4)
    a_ref = E * (c.q[sp] / c.m[sp])[:, None]
    with U.Context(n, c.q, c.m, leaf_cap=leaf_cap, precision=prec) as ctx:
        ctx.set_state(pos, vel, sp)
        acc, ph = ctx.tree_force(theta, eps)
        gp, gm = ctx.get_counts()
        ctx.step(1e-4, 2, 2, theta, eps)       # the electrons alone, then every particle
        p1, _ = ctx.get_state()
    assert rel_rms(acc, a_ref) <= tol and rel_rms(ph, phi) <= tol
    assert np.count_nonzero((gp != npp) | (gm != nmp)) <= 2 + n // 1000
    p_ref, _, _ = orc.run(pos, vel, sp, c.q, c.m, 1e-4, 2, 1, theta, eps, leaf_cap=leaf_cap,
                          nthreads=4)
    assert np.abs(p1 - p_ref).max() <= 1e-6 * np.abs(pos).max()


def test_pair_potential_over_the_range(U):
    """The FP64 walk's reciprocal square root at the ends of its own range and beyond: two
    particles a known distance apart, 240 pairs as an ensemble.  r^2 is exact, so phi is
    within an ulp of the charge over the distance, and the field three roundings more."""
    rng = np.random.default_rng(3)
    d = np.ldexp(rng.integers(1 << 19, 1 << 20, 240) / float(1 << 20), rng.integers(-60, 80, 240))
    d[:8] = np.ldexp(1.0, [-31, -30, -29, 49, 50, 51, 0, 1])
    m = len(d)
    pos = np.zeros((2 * m, 3))
    pos[1::2, 0] = d
    sp = np.tile(np.array([0, 1], dtype=np.int8), m)
    with U.Context(2 * m, (1.0, -1.0), (1.0, 1.0), leaf_cap=1, precision=0, sizes=[2] * m) as ctx:
        ctx.set_state(pos, np.zeros_like(pos), sp)
        acc, phi = ctx.tree_force(0.0, 0.0)
    u = np.spacing(1.0 / d)
    assert (np.abs(phi[0::2] + 1.0 / d) <= u).all() and (np.abs(phi[1::2] - 1.0 / d) <= u).all()
    f = 1.0 / (d * d)
    assert (np.abs(acc[0::2, 0] - f) <= 6 * np.spacing(f)).all()
    assert (np.abs(acc[1::2, 0] + f) <= 6 * np.spacing(f)).all()
