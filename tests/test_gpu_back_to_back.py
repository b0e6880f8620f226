"""Launches, and a warp's work items, that follow one another without a gap, bit for bit
against the plain half-step kernels (which form every value by the same
operations)."""
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


def run(D, prob, psi, steps, flags=0, plan=None):
    with D.Sim(prob, D.FP32, flags=flags) as s:
        if plan:
            s.set_plan(**plan)
        s.set_spinor(psi)
        s.step(steps)
        return s.get_spinor()


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("step", [False, True])
def test_many_strip_items_per_warp_with_a_moving_wave(D, axis, step):
    """Items of one row: 21 or 22 strips x 601 rows are more than five items for every warp the GPU
    holds at once.  67 steps: three link tables, and a pass of one step at the end."""
    N = (600, 601)
    k = [0.0, 0.0, 0.0]
    k[axis] = 2 * math.pi * 3 / N[axis]
    f = W.Fields(q=1.0, Apw_amp=0.5, Apw_k=tuple(k), Apw_omega=0.4, Apw_pol=1 - axis,
                 **(dict(step_axis=0, step_x0=N[0] / 2 + 0.25, step_V=0.3) if step else {}))
    prob = W.Problem(2, (N[0], N[1], 1), (1.0, 1.0, 1.0), 0.6, 0.4, f)
    psi = W.random_state(prob, 17)
    out = run(D, prob, psi, 67, plan=dict(chunk=1, two_step=1, chunk2=1))
    assert np.array_equal(out, run(D, prob, psi, 67, flags=D.FLAG_REFERENCE_KERNELS))


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("dims,N", [(2, (700, 300, 1)), (3, (96, 84, 40)), (3, (40, 36, 160))])
@pytest.mark.parametrize("field", ["free", "wave", "softcore"])
def test_hundreds_of_launches_over_a_state_in_cache(D, monkeypatch, graphs, dims, N, field):
    """A step starts while the blocks of the one before still write what it reads."""
    if not graphs:
        monkeypatch.setenv("DIRAC_NO_GRAPHS", "1")
    k = [0.0, 0.0, 0.0]
    k[dims - 1] = 2 * math.pi / N[dims - 1]
    f = {"free": {}, "wave": dict(q=1.0, Apw_amp=0.5, Apw_k=tuple(k), Apw_omega=0.3, Apw_pol=0),
         "softcore": dict(sc_Z=1.0, sc_a=1.0, sc_center=tuple(n / 2 for n in N))}[field]
    prob = W.Problem(dims, N, (1.0, 1.0, 1.0), 0.9 * W.stability_limit(dims), 0.4, W.Fields(**f))
    psi = W.random_state(prob, 23)
    assert np.array_equal(run(D, prob, psi, 401), run(D, prob, psi, 401, flags=D.FLAG_REFERENCE_KERNELS))


@pytest.mark.parametrize("n", [129, 194, 260])
@pytest.mark.parametrize("N", [(40, 200), (24, 2800)])
def test_graph_replays_with_link_tables(D, N, n):
    """A plane wave that does not move: its link tables are formed inside the graphs of 64 steps,
    and whatever their number the passes alone decide where the state ends up."""
    f = W.Fields(q=1.0, Apw_amp=0.5, Apw_k=(0.0, 2 * math.pi / N[1], 0.0), Apw_pol=0)
    prob = W.Problem(2, (N[0], N[1], 1), (1.0, 1.0, 1.0), 0.6, 0.4, f)
    psi = W.random_state(prob, 29)
    assert np.array_equal(run(D, prob, psi, n), run(D, prob, psi, n, flags=D.FLAG_REFERENCE_KERNELS))
