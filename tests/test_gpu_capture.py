"""A force call captured by the caller: the tree is built before the capture, so that its
records are still as the build left them when the captured walk first runs, and the graph
is replayed, also around calls that run at once.  Every pass gives the same bits."""
import numpy as np
import pytest

from paper_0709_3331_gb300.inputs import gaussian_cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,leaf_cap", [(500, 1), (2000, 16), (20001, 32)])
def test_captured_force_replays(prec, n, leaf_cap):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    c = gaussian_cloud(n + (n & 1), 1.0, 12)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        pos, vel, sp = (torch.tensor(np.ascontiguousarray(v[:n]), device="cuda")
                        for v in (c.pos, c.vel, c.species))
        acc, phi = torch.empty_like(pos), torch.empty_like(pos[:, 0])
        ref, ref_phi = torch.empty_like(acc), torch.empty_like(phi)
        with P.Context(n, c.q, c.m, leaf_cap=leaf_cap, precision=prec, stream=s.cuda_stream) as ctx:
            ctx.set_state(pos, vel, sp)
            ctx.tree_force(0.5, 0.01, ref, ref_phi)
            ctx.set_state(pos, vel, sp)
            ctx.tree_build()
            s.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
                ctx.tree_force(0.5, 0.01, acc, phi)
            for at_once in (True, False, False, True, False):
                acc.zero_()
                phi.zero_()
                if at_once:
                    ctx.tree_force(0.5, 0.01, acc, phi)
                else:
                    g.replay()
                s.synchronize()
                assert torch.equal(acc, ref) and torch.equal(phi, ref_phi)
            del g
