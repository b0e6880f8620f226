"""What FP64 simulations hold on the device."""
import numpy as np
import pytest

from paper_1309_3452_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SLACK = 64 << 20  # allocations come in pages of 2 MiB


@pytest.fixture(scope="module")
def D():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_3452_gb300 import dirac
    return dirac


def held(D, prob):
    """Bytes a simulation holds once it is made."""
    import torch
    with D.Sim(prob, D.FP64):  # (what the library allocates once)
        pass
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with D.Sim(prob, D.FP64):
        return free0 - torch.cuda.mem_get_info()[0]


def test_link_integrals_take_16_bytes_per_axis_and_value(D):
    prob = W.Problem(3, (128, 128, 64), (1.0, 1.0, 1.0), 0.5, 0.4)
    values = prob.n_planes * 128 * 128 * 64
    prob = prob.with_fields(q=1.0, A_links=np.full((3,) + tuple(prob.shape), 0.1))
    assert held(D, prob) <= D.state_bytes(3, prob.N, D.FP64) + 16 * 3 * values + SLACK
