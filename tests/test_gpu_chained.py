"""Runs of several substeps, whose kernels are launched as dependents of one another, against
the same substeps one call at a time and against captured blocks: the same state bit for
bit, from one particle to several waves of blocks."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,sizes", [(1, None), (2, None), (257, None), (4101, None),
                                     (60000, None), (900, [300, 1, 599])])
def test_chained_run(prec, n, sizes):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(n + (n & 1), 1.0, 7 + n)
    pos, vel, sp = c.pos[:n].copy(), c.vel[:n].copy(), c.species[:n].copy()
    out = []
    for mode in ("one call", "single substeps", "captured"):
        with P.Context(n, c.q, c.m, leaf_cap=16, precision=prec, sizes=sizes) as ctx:
            ctx.set_state(pos, vel, sp)
            if mode == "captured":
                ctx.set_graphs(True)
            for _ in range(6 if mode == "single substeps" else 1):
                ctx.step(1e-3, 1, 1 if mode == "single substeps" else 6, 0.5, 0.05)
            out.append(ctx.get_state() + ctx.tree_force(0.5, 0.05))
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)
