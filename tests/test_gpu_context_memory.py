"""What an FP32C context takes of the device, per particle of a system of 1,048,576: box
tables for the largest tree it can need (leaves of 1: 14 boxes of 296 bytes to a particle)
and the particles' own 700 bytes."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf_cap,most", [(1, 5514), (32, 1616)])
def test_bytes_per_particle(leaf_cap, most):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0709_3331_gb300 as P
    n = 1 << 20
    torch.zeros(1, device="cuda")
    before = torch.cuda.mem_get_info()[0]
    with P.Context(n, (1.0, -1.0), (1000.0, 1.0), leaf_cap=leaf_cap, precision=1):
        used = before - torch.cuda.mem_get_info()[0]
    assert used <= most * n
