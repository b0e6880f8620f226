"""The (2+1)D strip kernels where they can go wrong: grids around the 28 and 30
interior lanes of a strip and the smallest row counts (three rows take one
step per pass, four and more two), a Klein step inside, at the edge of and
outside a strip, moving plane waves along either axis (one link table per step
of a pass), isotropic and not.  The plain half-step kernels form every value
by the same operations, so the states agree bit for bit."""
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


def fields(name, N):
    wave = dict(q=1.0, Apw_amp=0.5, Apw_omega=0.4)
    return {"step_mid": W.Fields(step_axis=0, step_x0=N[0] / 2 + 0.25, step_V=0.7),
            "step_edge": W.Fields(step_axis=0, step_x0=27.75, step_V=0.7),
            "step_first": W.Fields(step_axis=0, step_x0=0.0, step_V=-0.5),
            "step_y": W.Fields(step_axis=1, step_x0=1.25, step_V=0.7),
            "step_const": W.Fields(step_axis=0, step_x0=N[0] / 3 + 0.25, step_V=0.7, q=1.0, A_const=(0.2, 0.1, 0.0)),
            "wave_y": W.Fields(**wave, Apw_k=(0.0, 2 * math.pi / N[1], 0.0), Apw_pol=0),
            "wave_x": W.Fields(**wave, Apw_k=(2 * math.pi / N[0], 0.0, 0.0), Apw_pol=1),
            "wave_step": W.Fields(**wave, Apw_k=(0.0, 2 * math.pi / N[1], 0.0), Apw_pol=0, step_axis=0,
                                  step_x0=N[0] / 2 + 0.25, step_V=0.3)}[name]


@pytest.mark.parametrize("N", [(27, 3), (28, 4), (29, 5), (57, 9), (61, 64)])
@pytest.mark.parametrize("name", ["step_mid", "step_edge", "step_first", "step_y", "step_const", "wave_y", "wave_x",
                                  "wave_step"])
@pytest.mark.parametrize("dy", [1.0, 1.2])
def test_strips_equal_the_plain_kernels_bitwise(D, N, name, dy):
    prob = W.Problem(2, (N[0], N[1], 1), (1.0, dy, 1.0), 0.6, 0.4, fields(name, N))
    psi = W.random_state(prob, 31)
    out = []
    for flags in (0, D.FLAG_REFERENCE_KERNELS):
        with D.Sim(prob, D.FP32, flags=flags) as s:
            s.time = 0.2
            s.set_spinor(psi)
            s.step(7)
            s.step(4)
            out.append(s.get_spinor())
    assert np.array_equal(out[0], out[1])
