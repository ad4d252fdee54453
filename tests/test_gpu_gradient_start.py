"""The gradient of a run from the current state does not depend on the calls before it: a
force call and a run of steps store accelerations, which in FP32C contexts are another
walk's than the gradient's forward run takes.  Its final state is that of a context which
was given the same state, bit for bit, and so are its loss and, but for the order of the
adjoint's atomic sums, its gradients."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu

DT, K, STEPS, THETA, EPS = 1e-3, 5, 20, 0.5, 0.01


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("before", ["force", "step", "energy"])
@pytest.mark.parametrize("n,checkpoint", [(3000, 5), (3000, 20), (20000, 10)])
def test_gradient_after_other_calls(prec, before, n, checkpoint):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(n, 1.5, 31)
    start = (c.pos, c.vel)
    out = []
    for other in (True, False):
        with P.Context(n, c.q, c.m, leaf_cap=16, precision=prec) as ctx:
            ctx.set_state(*start, c.species)
            if other:
                if before == "force":
                    ctx.tree_force(THETA, EPS)
                elif before == "step":
                    ctx.step(DT, K, K, THETA, EPS)
                    start = ctx.get_state()
                else:
                    ctx.energy(THETA, EPS)
            grad = ctx.grad_ke_electrons(DT, K, STEPS, THETA, EPS, checkpoint)
            out.append((grad, ctx.get_state()))
    ((l0, gx0, gv0), (p0, v0)), ((l1, gx1, gv1), (p1, v1)) = out
    assert np.array_equal(p0, p1) and np.array_equal(v0, v1) and l0 == l1
    # the adjoint's sums in any order, about 1e3 terms: of the pairs in FP64 (1e3 x 1e-16, and
    # its growth over the run by 1e3), of the boxes of FP32C contexts in FP32 (35 x 6e-8 of
    # the far field's part)
    tol = 1e-10 if prec == 0 else 1e-5
    assert np.abs(gx0 - gx1).max() <= tol * np.abs(gx0).max()
    assert np.abs(gv0 - gv1).max() <= tol * np.abs(gv0).max()


def test_step_after_a_gradient_is_an_ordinary_step():
    """The other way round: a step after the gradient does not start from its walk's."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(3000, 1.5, 32)
    with P.Context(c.n, c.q, c.m, leaf_cap=16, precision=1) as ctx:
        ctx.set_state(c.pos, c.vel, c.species)
        ctx.grad_ke_electrons(DT, K, K, THETA, EPS, K)
        mid = ctx.get_state()
        ctx.step(DT, K, K, THETA, EPS)
        a = ctx.get_state()
        ctx.set_state(*mid, c.species)
        ctx.step(DT, K, K, THETA, EPS)
        b = ctx.get_state()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
