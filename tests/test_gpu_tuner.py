"""The launch-shape tuner times the kernels that have shapes: on a small ring, whose few limbs run by other routes, it launches
what it launches on a ring without those routes, and the routes are back afterwards."""
import pytest

from paper_2606_10477_gb300 import hedap

pytestmark = pytest.mark.gpu


def launches_of_tune(log_n, alpha, n_p):
    g = hedap.Context(log_n, [45] * 6, [60] * n_p, alpha, 40.0, 64, 1)
    n = hedap.launch_count()
    g.ntt_tune(4 * g.n_q, 1)
    return hedap.launch_count() - n, g


@pytest.mark.parametrize("log_n", [10, 12, 13])
@pytest.mark.parametrize("alpha,n_p", [(1, 1), (2, 2), (4, 5)])
def test_tuner_times_the_launch_shapes(log_n, alpha, n_p):
    import torch
    want, _ = launches_of_tune(14, alpha, n_p)
    got, g = launches_of_tune(log_n, alpha, n_p)
    assert got == want
    x = torch.zeros((2, g.n_q, g.N), dtype=torch.int64, device="cuda")
    n = hedap.launch_count()
    g.ntt_batch(x, g.n_q, 0)
    assert hedap.launch_count() - n == 1
    g.sync()
