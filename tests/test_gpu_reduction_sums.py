"""The reductions' sums over many cells per thread: as exact as FP64 sums of the
cells' terms, whatever the states' precision."""
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


@pytest.mark.parametrize("precision,flags", [("fp64", 0), ("fp32", 0), ("fp32", 2)])
def test_terms_of_three_magnitudes(D, precision, flags):
    """One value per cell, 1, 2^-12 or 2^-24, with exact squares; a thread meets the large ones first.
    A sum of 1, 2^-24 and fourteen 2^-48 is exact in FP64, and at most 64 roundings of 2^-53 follow
    one another on the way to the total."""
    rows = 80000  # 32 cells each: 16 for each of the (at most) 152 x 4 x 256 threads
    prob = W.Problem(2, (32, rows, 1), (1.0, 1.0, 1.0), 0.6, 0.4)
    v = np.full(rows, 2.0 ** -24)
    v[:2 * 4864] = 2.0 ** -12
    v[:4864] = 1.0
    psi = np.zeros(prob.shape, dtype=np.complex128)
    psi[0, 0] = v[:, None]
    total = 32 * math.fsum(v * v)
    tol = 64 * 2.0 ** -53 * total
    with D.Sim(prob, D.FP64 if precision == "fp64" else D.FP32, flags=flags) as s:
        s.set_spinor(psi)
        E, naive = s.norm()
        assert abs(naive - total) <= tol and abs(E - total) <= tol
        assert abs(s.partial_density(0, -1.0) - total) <= tol


@pytest.mark.parametrize("flags", [0, 2])
def test_sums_beyond_the_floats_range(D, flags):
    """Squares that a float holds and their sums do not, and an infinite and a NaN value in one cell."""
    prob = W.Problem(2, (32, 80000, 1), (1.0, 1.0, 1.0), 0.6, 0.4)
    psi = np.zeros(prob.shape, dtype=np.complex128)
    v = float(np.float32(1.5e19))
    psi[0] = v
    n = psi[0].size
    with D.Sim(prob, D.FP32, flags=flags) as s:
        s.set_spinor(psi)
        _, naive = s.norm()
        # every square is rounded once, to 2^-24 of itself
        assert abs(naive - n * v * v) <= 2.0 ** -24 * n * v * v
        for bad in (np.inf, np.nan):
            psi[0, 0, 41234, 7] = bad
            s.set_spinor(psi)
            n = s.partial_density(0, -1.0)
            assert np.isinf(n) and n > 0 if np.isinf(bad) else np.isnan(n)
            with pytest.raises(D.DiracError):  # a functional that is not finite is reported
                s.norm()
