"""hedap_launch_count is the number of kernels launched: one for a transform whose limbs each fit a thread-block cluster (small
rings, up to 2^21 words), two otherwise."""
import pytest

from paper_2606_10477_gb300 import hedap

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("log_n,polys,launches", [(10, 1, 1), (10, 600, 2), (13, 64, 1), (13, 65, 2), (14, 1, 2)])
@pytest.mark.parametrize("inverse", [False, True])
def test_launches_of_one_transform(log_n, polys, launches, inverse):
    import torch
    g = hedap.Context(log_n, [45, 45, 45], [60], 1, 30.0, 0, 1)  # 4 limbs a polynomial
    x = torch.zeros((polys, 4, g.N), dtype=torch.int64, device="cuda")
    n = hedap.launch_count()
    g.ntt_batch(x, 4, 0, inverse=inverse)
    assert hedap.launch_count() - n == launches
    g.sync()
