"""Absorbing layers in the FP32 kernels, whose cells share coefficients where no
layer reaches: every link path, Klein steps inside, in a layer and at an edge,
a uniform imaginary part, layers on some axes only, as wide as the grid and
narrower than a cell.  The plain half-step kernels read one record per value;
the states agree bit for bit."""
import math

import numpy as np
import pytest

from paper_1309_3452_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 8


@pytest.fixture(scope="module")
def D():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1309_3452_gb300 import dirac
    return dirac


def fields(name, dims, N):
    layers = dict(abs_W=0.5, abs_width=3.0, abs_axes=(1 << dims) - 1)
    k = [0.0, 0.0, 0.0]
    k[dims - 1] = 2 * math.pi / N[dims - 1]
    wave = dict(q=1.0, Apw_amp=0.5, Apw_k=tuple(k), Apw_omega=0.4, Apw_pol=0)
    return {"plain": W.Fields(**layers), "v0_imag": W.Fields(**layers, V0=0.3, V0_imag=-0.2),
            "one_axis": W.Fields(abs_W=0.5, abs_width=2.5, abs_axes=1),
            "step": W.Fields(**layers, step_axis=dims - 1, step_x0=N[dims - 1] / 2 + 0.25, step_V=0.7),
            "step_x": W.Fields(**layers, step_axis=0, step_x0=N[0] / 2 + 0.25, step_V=0.7),
            "wave": W.Fields(**layers, **wave),
            "wave_step": W.Fields(**layers, **wave, step_axis=1, step_x0=N[1] / 2 + 0.25, step_V=0.7),
            "step_layer": W.Fields(**layers, step_axis=0, step_x0=1.25, step_V=0.7),
            "step_edge": W.Fields(**layers, step_axis=1, step_x0=N[1] - 3.0, step_V=0.7),
            "wave_x": W.Fields(**layers, q=1.0, Apw_amp=0.5, Apw_k=(2 * math.pi / N[0], 0.0, 0.0), Apw_omega=0.4,
                               Apw_pol=1),
            "const_a": W.Fields(**layers, q=1.0, A_const=(0.2, 0.1, 0.0)),
            "static_wave": W.Fields(**layers, q=1.0, Apw_amp=0.5, Apw_k=(0.3, 0.2, 0.0), Apw_pol=0),
            "wide": W.Fields(abs_W=0.5, abs_width=100.0, abs_axes=1),
            "narrow": W.Fields(abs_W=0.5, abs_width=0.25, abs_axes=(1 << dims) - 1)}[name]


@pytest.mark.parametrize("dims,N", [(2, (29, 5, 1)), (2, (57, 9, 1)), (2, (64, 3, 1)), (3, (33, 26, 5)),
                                    (3, (31, 29, 4)), (3, (40, 57, 3))])
@pytest.mark.parametrize("name", ["plain", "v0_imag", "one_axis", "step", "step_x", "wave", "wave_step",
                                  "step_layer", "step_edge", "wave_x", "const_a", "static_wave", "wide", "narrow"])
@pytest.mark.parametrize("dy", [1.0, 1.2])
def test_layers_against_the_plain_kernels_and_fp64(D, dims, N, name, dy):
    prob = W.Problem(dims, N, (1.0, dy, 1.0), 0.9 * W.stability_limit(dims), 0.6, fields(name, dims, N))
    psi = W.random_state(prob, 41)
    out = []
    for precision, flags in ((D.FP32, 0), (D.FP32, D.FLAG_REFERENCE_KERNELS), (D.FP64, 0)):
        with D.Sim(prob, precision, flags=flags) as s:
            s.set_spinor(psi)
            s.step(STEPS - 1)
            s.step(1)  # a call's last step runs the kernels that accumulate the functional
            out.append(s.get_spinor())
    # (a plane wave along x in (3+1)D: the fused kernels form its links per site,
    # the plain ones from a table of the shared factor)
    assert np.array_equal(out[0], out[1]) or (dims == 3 and name == "wave_x")
    # each half-step rounds a value formed from terms of at most a few times the
    # state's largest magnitude a dozen times
    top = np.abs(psi).max()
    assert np.abs(out[0] - out[2]).max() <= 2 * STEPS * 16 * 2.0 ** -24 * top
