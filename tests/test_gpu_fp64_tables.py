"""FP64 runs with tabulated alpha and gamma (potentials that do not change in
time) in every combination with the link paths, on odd sizes, against the
oracle.  Tolerance: the parity tests' 1e-12 relative (rounding order only)."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_1309_3452_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_3452_gb300 import dirac
    return dirac


@pytest.mark.parametrize("dims,N", [(2, (33, 5, 1)), (3, (7, 33, 5))])
@pytest.mark.parametrize("coef", ["softcore", "layers", "static"])
@pytest.mark.parametrize("links", ["none", "const", "wave", "table"])
def test_fp64_tables(D, dims, N, coef, links):
    prob = W.Problem(dims, N, (1.0, 1.0, 1.0), 0.9 * W.stability_limit(dims), 0.4)
    k = [0.0, 0.0, 0.0]
    k[dims - 1] = 2 * math.pi / N[dims - 1]
    f = {"softcore": dict(sc_Z=1.2, sc_a=0.7, sc_center=(3.0, 2.5, 2.0)),
         "layers": dict(V0=0.1, abs_W=0.5, abs_width=2.0, abs_axes=(1 << dims) - 1),
         "static": dict(V_static=W.random_potential(prob, 5, 0.5))}[coef]
    f |= {"none": {}, "const": dict(q=0.8, A_const=(0.3, -0.2, 0.1)),
          "wave": dict(q=1.0, Apw_amp=0.4, Apw_k=tuple(k), Apw_omega=0.3, Apw_pol=0),
          "table": dict(q=1.0, A_links=W.random_links(prob, 6, 0.4))}[links]
    prob = prob.with_fields(**f)
    psi = W.random_state(prob, 8)
    ref = O.step(prob, psi, 20, 0.1)
    with D.Sim(prob, D.FP64) as s:
        s.time = 0.1
        s.set_spinor(psi)
        s.step(20)
        out = s.get_spinor()
    assert np.linalg.norm(out - ref) <= 1e-12 * np.linalg.norm(ref)
