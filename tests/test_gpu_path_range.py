"""Per-path records at the end of the index range: paths up to 2^32 - 1, in tasks of one path to several, are
the oracle's."""
import pytest

import workloads as W
from gpu_helpers import PathTally, gpu_problem, oracle_inputs, tolerances
from oracle import mc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_ACC64])
@pytest.mark.parametrize("n,short", [(1, 0), (31, 0), (64, 0), (2049, 0), (50, 1), (100, 32)])
def test_last_paths_match_oracle(n, short, precision):
    prob = W.c0_small_fp64().replace(precision=precision)
    x, y = W.identity_mesh(prob)
    _, inp, nodes = oracle_inputs(prob, x, y, prob.t0, 0)
    margin, value = tolerances(prob)
    begin = 2 ** 32 - short - n
    h = gpu_problem(prob)
    tally = PathTally()
    for m in (0, 17, len(nodes) - 1):
        gv, gs, gd = h.debug_paths(m, begin, n)
        ov, os_, od, mg = mc.paths(inp, m, int(nodes[m, 0]), int(nodes[m, 1]), begin, n)
        tally.add(gv, gs, gd, ov, os_, od, mg, margin, value)
    h.close()
    tally.check()
