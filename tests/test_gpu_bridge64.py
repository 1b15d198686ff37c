"""FP64 path decisions where the bridge test is decided in FP32 and left to FP64 only when unsure: exit
steps and sides of every path against the oracle (values within the growth of a rounding over 50 substeps,
(1 + 0.2)^50 1e-15, rounded up to 1e-10), with step sizes from ones that rarely reach the
boundary to ones whose crossing probabilities are near 1, both generator forms and starts next to a
side, in a corner and inside."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem, oracle_inputs
from oracle import mc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("dt", [1e-5, 1e-3, 1e-2, 0.3, 20.0])
def test_exit_decisions_match_oracle(dt, form):
    prob = W.c0_small_fp64().replace(nx=41, ny=37, px=4, py=3, dt=dt, form=form, tau=1.0 if form else 1e-2, substeps=50,
                                     monitor_params=[3.0, 6.0, 0.45, 0.55])
    x, y = W.identity_mesh(prob)
    om, inp, nodes = oracle_inputs(prob, x, y, prob.t0, 0)
    h = gpu_problem(prob)
    for m in (0, len(nodes) // 3, len(nodes) - 1):
        v, steps, side = h.debug_paths(m, 0, 3000)
        ov, osteps, oside, margin = mc.paths(inp, m, int(nodes[m, 0]), int(nodes[m, 1]), 0, 3000)
        clear = margin > 1e-12
        assert clear.mean() > 0.999
        assert np.array_equal(steps[clear], osteps[clear]) and np.array_equal(side[clear], oside[clear])
        assert np.abs(v - ov)[clear].max() <= 1e-10
    h.close()
