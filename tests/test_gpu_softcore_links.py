"""A soft core with tabulated static links in the FP32 kernels (one packed update
per component) against the plain half-step kernels, which form every value by
the same operations: the states agree bit for bit.  Ragged sizes around the
strips' 28 and 30 lanes and the tiles' 32 x 26 cells, with a Klein step,
isotropic and not."""
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


@pytest.mark.parametrize("dims,N", [(2, (29, 5, 1)), (2, (57, 64, 1)), (2, (64, 3, 1)), (3, (33, 26, 5)), (3, (31, 29, 9))])
@pytest.mark.parametrize("links", ["integrals", "wave"])
@pytest.mark.parametrize("step", [False, True])
@pytest.mark.parametrize("dy", [1.0, 1.2])
def test_against_the_plain_kernels(D, dims, N, links, step, dy):
    prob = W.Problem(dims, N, (1.0, dy, 1.0), 0.9 * W.stability_limit(dims), 0.6)
    f = dict(sc_Z=1.1, sc_a=0.8, sc_center=(N[0] / 2, N[1] / 2, N[2] / 2 if dims == 3 else 0.0), V0=0.1, q=1.0)
    f |= dict(A_links=W.random_links(prob, 6, 0.4)) if links == "integrals" else \
        dict(Apw_amp=0.5, Apw_k=(0.3, 0.2, 0.0), Apw_pol=0)
    if step:
        f |= dict(step_axis=0, step_x0=N[0] / 2 + 0.25, step_V=0.7)
    prob = prob.with_fields(**f)
    psi = W.random_state(prob, 43)
    out = []
    for flags in (0, D.FLAG_REFERENCE_KERNELS):
        with D.Sim(prob, D.FP32, flags=flags) as s:
            s.set_spinor(psi)
            s.step(7)
            s.step(1)  # a call's last step runs the kernels that accumulate the functional
            E = s.norm()[0]
            out.append((s.get_spinor(), E))
    assert np.array_equal(out[0][0], out[1][0])
    # the functional accumulated by the step: FP32 terms, each rounded a few times
    assert abs(out[0][1] - out[1][1]) <= 1e-6
