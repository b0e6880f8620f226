"""The fused (3+1)D kernels' two tile heights and the quad state layout at the
sizes where they can go wrong: rows around the tiles' 26 and 28 interior rows
(one tile exactly full, one row over, the smallest remainder), columns around
the 32 interior columns, and field paths with per-cell tables.  Every value is
formed by the same operations in the same order as in the plain half-step
kernels (planar layout, one value at a time), so the two must agree bit for
bit, whichever tile runs."""
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
    kz = 2 * math.pi / N[2]
    c = tuple(n / 2.0 for n in N)
    soft = dict(sc_Z=1.0, sc_a=1.0, sc_center=c)
    wave = dict(q=1.0, Apw_amp=0.5, Apw_k=(0.0, 0.0, kz), Apw_omega=kz, Apw_pol=0)
    return {"free": W.Fields(), "klein": W.Fields(step_axis=1, step_x0=N[1] / 2 + 0.25, step_V=0.7),
            "const_a": W.Fields(q=1.0, A_const=(0.2, -0.3, 0.1)), "laser": W.Fields(**soft, **wave),
            "layers": W.Fields(abs_W=0.5, abs_width=3.0, abs_axes=7)}[name]


@pytest.mark.parametrize("N", [(33, 26, 5), (31, 28, 4), (32, 29, 3), (65, 53, 4), (2, 57, 6), (40, 84, 3)])
@pytest.mark.parametrize("name", ["free", "klein", "const_a", "laser", "layers"])
def test_tiles_equal_the_plain_kernels_bitwise(D, N, name):
    prob = W.Problem(3, N, (1.0, 1.0, 1.0), 0.9 * W.stability_limit(3), 0.6, fields(name, N))
    psi = W.random_state(prob, 23)
    out = []
    for flags in (0, D.FLAG_REFERENCE_KERNELS):
        with D.Sim(prob, D.FP32, flags=flags) as s:
            s.set_spinor(psi)
            s.step(5)
            s.step(1)  # a call's last step runs the kernels that accumulate the functional
            out.append(s.get_spinor())
    assert np.array_equal(out[0], out[1])
