"""The functional's cross terms where the vector potential turns the neighbours
into one another (a pure gauge): the rotated differences nearly vanish, so what
a rotation rounds off relative to the neighbours shows.

Tolerance, with the naive norm as the unit: a rotated difference is formed from
four products of about one with an error of at most 8 x 2^-48 each, below 2^-43
for all of a cell's terms beside its values; the differences themselves are of
the size of the state's rounding, 2^-23, and their own roundings 2^-24 of that;
the sums are FP64's.  2^-42 in all."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_1309_3452_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -42


@pytest.fixture(scope="module")
def D():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_3452_gb300 import dirac
    return dirac


def check(D, prob, psi, precision, flags):
    psi = psi.astype(np.complex64).astype(np.complex128)
    ref = O.observables(prob, psi, 0.0)
    with D.Sim(prob, D.FP64 if precision == "fp64" else D.FP32, flags=flags) as s:
        s.set_spinor(psi)
        E, naive = s.norm()
    assert abs((E - naive) - (ref["E"] - ref["naive"])) <= TOL * ref["naive"]


def problem(dims, N):
    return W.Problem(dims, N, (1.0, 1.1, 0.9) if dims == 3 else (1.0, 1.1, 1.0), 0.5, 0.4)


@pytest.mark.parametrize("precision,flags", [("fp64", 0), ("fp32", 0), ("fp32", 2)])
@pytest.mark.parametrize("dims,N", [(2, (31, 9, 1)), (2, (65, 70, 1)), (3, (33, 9, 7)), (3, (32, 12, 10))])
def test_static_links(D, dims, N, precision, flags):
    prob = problem(dims, N)
    chi = np.random.default_rng(4).uniform(-math.pi, math.pi, size=(2 * N[2], 2 * N[1], 2 * N[0]))

    def at(H):
        return chi[H[2], H[1], H[0]]
    prob = prob.with_fields(q=1.0, A_links=W.link_integrals(prob, lambda a, S, E: at(E) - at(S)))
    psi = np.stack([np.exp(1j * at(W.half_lattice_points(prob, p))) for p in range(prob.n_planes)])
    check(D, prob, psi, precision, flags)


@pytest.mark.parametrize("precision,flags", [("fp64", 0), ("fp32", 0), ("fp32", 2)])
@pytest.mark.parametrize("dims,N,along,pol", [(2, (31, 9, 1), 1, 0), (2, (65, 70, 1), 0, 1), (3, (33, 9, 7), 2, 0),
                                              (3, (32, 12, 10), 0, 1), (3, (33, 9, 10), 1, 2)])
def test_plane_wave(D, dims, N, along, pol, precision, flags):
    """A wave so long that its phase is the same everywhere, 2 pi j over the period of the axis."""
    prob = problem(dims, N)
    phi = 2 * math.pi * max(1, N[pol] // 6) / (2 * N[pol])
    k = [0.0, 0.0, 0.0]
    k[along] = 1e-12
    prob = prob.with_fields(q=1.0, Apw_amp=phi / (0.5 * prob.dx[pol]), Apw_k=tuple(k), Apw_pol=pol)
    psi = np.stack([np.exp(1j * phi * W.half_lattice_points(prob, p)[pol]) for p in range(prob.n_planes)])
    check(D, prob, psi, precision, flags)
