"""The plane waves' link tables on grids long along the wave."""
import math

import numpy as np
import pytest

from paper_1309_3452_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_3452_gb300 import dirac
    return dirac


def problem(N):
    return W.Problem(2, N, (1.0, 1.0, 1.0), 0.6, 0.4,
                     W.Fields(q=1.0, Apw_amp=0.5, Apw_k=(2 * math.pi * 1000 / N[0], 0.0, 0.0), Apw_omega=0.4, Apw_pol=1))


def test_2_to_the_31_table_entries(D):
    """32 steps of 2 x 2^25 entries: one call's tables, and those of one step at a time, give the same state."""
    import torch
    prob = problem((1 << 24, 2, 1))
    torch.manual_seed(3)
    psi = torch.randn((4, 2, 1 << 24), dtype=torch.complex128, device="cuda")
    out = []
    for calls, n in ((1, 32), (32, 1)):
        with D.Sim(prob, D.FP64) as s:
            s.set_spinor_device(psi.data_ptr())
            for _ in range(calls):
                s.step(n)
            out.append(torch.empty_like(psi))
            s.get_spinor_device(out[-1].data_ptr())
            torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])


def test_memory_of_a_grid_long_along_the_wave(D):
    """One step's factors (256 bytes per cell along the wave) where a quarter of the state holds no more."""
    import torch
    prob = problem((1 << 20, 8, 1))
    with D.Sim(prob, D.FP32) as s:  # (whatever the library allocates once)
        pass
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    with D.Sim(prob, D.FP32) as s:
        used = free0 - torch.cuda.mem_get_info()[0]
    assert used <= D.state_bytes(2, prob.N, D.FP32) + (256 << 20) + (64 << 20)  # (allocations come in 2 MiB pages)


@pytest.mark.parametrize("N", [(40000, 8), (20000, 5), (70000, 4), (2500, 9)])
def test_tables_of_fewer_steps(D, N):
    """1, 2 and 26 steps per table; 67 steps, so that tables, passes and calls end at different steps."""
    prob = problem((N[0], N[1], 1))
    psi = W.random_state(prob, 37)
    out = []
    for flags in (0, D.FLAG_REFERENCE_KERNELS):
        with D.Sim(prob, D.FP32, flags=flags) as s:
            s.set_spinor(psi)
            s.step(40)
            s.step(27)
            out.append(s.get_spinor())
    assert np.array_equal(out[0], out[1])
