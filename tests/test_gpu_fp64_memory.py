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


@pytest.mark.parametrize("field", ["softcore", "static"])
def test_coefficient_tables_make_room(D, field):
    """As many simulations as their states (and static arrays) alone would let fit, to four; those whose
    tables go keep their values, also one that another thread steps meanwhile."""
    import threading
    import torch
    N = (128, 128, 64)
    prob = W.Problem(3, N, (1.0, 1.0, 1.0), 0.5, 0.4)
    f = {"softcore": dict(sc_Z=1.0, sc_a=1.0, sc_center=(64.0, 64.0, 32.0)),
         "static": dict(V_static=W.random_potential(prob, 5, 0.5))}[field]
    prob = prob.with_fields(**f)
    own = D.state_bytes(3, N, D.FP64) + (8 * prob.n_planes * N[0] * N[1] * N[2] if field == "static" else 0)
    torch.manual_seed(1)
    psi = torch.randn((8, 64, 128, 128), dtype=torch.complex128, device="cuda")
    out = torch.empty_like(psi)

    def state(s):
        s.get_spinor_device(out.data_ptr())
        torch.cuda.synchronize()
        return out.clone()

    with D.Sim(prob, D.FP64) as s:
        s.set_spinor_device(psi.data_ptr())
        for _ in range(4):  # (graphs of 64 steps)
            s.step(70)
        want = state(s)
    torch.cuda.synchronize()
    room = 3 << 30
    fill = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    sims = []
    try:
        stream = torch.cuda.Stream()
        sims = [D.Sim(prob, D.FP64), D.Sim(prob, D.FP64, stream=stream.cuda_stream)]
        for s in sims:
            s.set_spinor_device(psi.data_ptr())
            s.step(70)
        bytes_before = sims[0].algorithmic_bytes
        torch.cuda.synchronize()
        t = threading.Thread(target=lambda: [sims[1].step(70) for _ in range(3)])
        t.start()
        with pytest.raises(D.DiracError) as e:
            while len(sims) < 64:
                sims.append(D.Sim(prob, D.FP64))
        t.join()
        assert e.value.status == D.ERR_OOM
        assert len(sims) >= room // own - 4
        assert sims[0].algorithmic_bytes == bytes_before
        for _ in range(3):
            sims[0].step(70)
        for s in sims[2:]:
            s.close()
        for s in sims[:2]:
            assert torch.equal(state(s), want)
    finally:
        for s in sims:
            s.close()
        del fill
        torch.cuda.empty_cache()
