"""Round plan and reduction at the edges of their blocks: 4096 nodes planned at a time, two or eight nodes
reduced by a block (two up to 2432).  Tolerance 1e-10 as for all FP64 estimates: sums of at most 4097 values of
order 1 regrouped are within 4097 * 2^-53 of each other.  Standard errors have no such bound (where all paths
of a node end at one value they are the root of a rounding); they are compared bitwise, a served request's with
the problem's alone, which come from different kernels."""
import time

import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem, oracle_inputs
from oracle import mc
from test_gpu_serving import alone, server_params, submit

pytestmark = pytest.mark.gpu


def line(M, **kw):
    """One horizontal interface line of M nodes."""
    return W.c0_small_fp64().replace(nx=M + 2, ny=5, px=1, py=2, substeps=1, **kw)


@pytest.mark.parametrize("M", [1, 2, 3, 15, 16, 17, 31, 33, 2431, 2432, 2433, 4095, 4096, 4097, 9000])
@pytest.mark.parametrize("se_target", [0.0, 2e-3])
def test_nodes_match_oracle(M, se_target):
    prob = line(M, paths_per_node=33, se_target=se_target, max_paths_per_node=4097 if se_target else 0)
    x, y = W.identity_mesh(prob)
    om, inp, nodes = oracle_inputs(prob, x, y, prob.t0, 0)
    oest, ose, on, osteps = mc.interface_mc(prob, x, y, om, nodes, 0, np.float64)
    h = gpu_problem(prob)
    est, se, n, _ = h.interface_mc()
    st = h.stats()
    h.close()
    assert len(nodes) == M and np.array_equal(n, on)
    assert st["paths"] == on.sum() and st["path_steps"] == osteps.sum() and st["max_se"] == se.max()
    assert np.abs(est - oest).max() <= 1e-10


def test_capped_rounds_over_several_passes():
    """6000 nodes of one task each, 4500 tasks a round: the cap falls into the second pass."""
    import torch

    import paper_1504_00084_gb300 as S
    probs = [line(3000, paths_per_node=33, seed=k) for k in (1, 2)]
    refs = [alone(p) for p in probs]
    q = server_params(W.PREC_FP64, 33, 0.0, 0, round_paths=4500 * 2048)
    q.max_nodes = 1 << 14
    with S.SddServer(q, torch.cuda.Stream()) as srv:
        ids = [submit(srv, p) for p in probs]
        done = []
        for _ in range(20000):  # the solves of such long strips take a while
            srv.progress()
            done += srv.poll()
            if len(done) == 2:
                break
            time.sleep(1e-3)
        assert len(done) == 2
        for rid, (rx, ry, rest, rse) in zip(ids, refs):
            out = srv.result(rid)
            assert np.array_equal(out["x"], rx) and np.array_equal(out["y"], ry)
            assert np.array_equal(out["est"], rest) and np.array_equal(out["se"], rse)
