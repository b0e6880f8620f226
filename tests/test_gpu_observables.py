"""The reductions (functional, naive norm, partial density) of a state just
set, against the oracle, at row lengths around the 32 cells of a warp's piece
and for every link path: none, constant, a plane wave along each axis,
tabulated links.

Tolerances: FP64 states differ from the oracle by the order of sums of at most
8 * 33 * 9 * 7 values, 1e-13 relative.  FP32 states round every value once
(2^-24 relative), so every |v|^2 and every cross term by at most 2^-23 plus
the few roundings of its own products: 1e-6 of the naive norm."""
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


def wave(N, axis):
    k = [0.0, 0.0, 0.0]
    k[axis] = 2 * math.pi / N[axis]
    return dict(q=1.0, Apw_amp=0.5, Apw_k=tuple(k), Apw_omega=0.3, Apw_phase=0.2, Apw_pol=1 if axis == 0 else 0)


@pytest.mark.parametrize("dims,N", [(2, (31, 9, 1)), (2, (33, 2, 1)), (3, (32, 5, 4)), (3, (33, 9, 7)), (3, (2, 3, 2))])
@pytest.mark.parametrize("links", ["none", "const", "wave_x", "wave_last", "table"])
@pytest.mark.parametrize("precision,flags", [("fp64", 0), ("fp32", 0), ("fp32", 2)])
def test_reductions_of_a_set_state(D, dims, N, links, precision, flags):
    prob = W.Problem(dims, N, (1.0, 1.1, 0.9) if dims == 3 else (1.0, 1.1, 1.0), 0.5, 0.4)
    f = {"none": {}, "const": dict(q=0.7, A_const=(0.2, -0.3, 0.1)), "wave_x": wave(N, 0),
         "wave_last": wave(N, dims - 1), "table": dict(q=1.0, A_links=W.random_links(prob, 3, 0.4))}[links]
    prob = prob.with_fields(**f)
    psi = W.random_state(prob, 9)
    t = 0.35
    ref = O.observables(prob, psi, t)
    x = [W.site_positions(prob, p)[0] for p in range(prob.n_planes)]
    dens = sum(float(np.sum(np.abs(psi[p][x[p] > N[0] / 2 - 0.3]) ** 2)) for p in range(prob.n_planes))
    tol = (1e-13 if precision == "fp64" else 1e-6) * ref["naive"]
    with D.Sim(prob, D.FP64 if precision == "fp64" else D.FP32, flags=flags) as s:
        s.time = t
        s.set_spinor(psi)
        E, naive = s.norm()
        assert abs(E - ref["E"]) <= tol and abs(naive - ref["naive"]) <= tol
        assert abs(s.partial_density(0, N[0] / 2 - 0.3) - dens) <= tol
