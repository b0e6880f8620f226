"""Simulations made on a stream that is not ordered after the legacy stream:
their tables are there when the first kernel of that stream reads them."""
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


@pytest.mark.parametrize("dims,N", [(2, (257, 130, 1)), (3, (65, 40, 33))])
@pytest.mark.parametrize("field", ["layers", "softcore"])
def test_tables_on_a_non_blocking_stream(D, dims, N, field):
    import torch
    f = {"layers": dict(V0=0.1, abs_W=0.5, abs_width=4.0, abs_axes=(1 << dims) - 1),
         "softcore": dict(sc_Z=1.0, sc_a=1.0, sc_center=tuple(n / 2 for n in N))}[field]
    prob = W.Problem(dims, N, (1.0, 1.0, 1.0), 0.9 * W.stability_limit(dims), 0.4, W.Fields(**f))
    psi = W.random_state(prob, 5)
    out = []
    for stream in (torch.cuda.default_stream(), torch.cuda.Stream()):
        for _ in range(4):
            with D.Sim(prob, D.FP32, stream=stream.cuda_stream) as s:
                s.set_spinor(psi)
                s.step(5)
                out.append(s.get_spinor())
    for o in out[1:]:
        assert np.array_equal(o, out[0])
