"""FP32 problems whose switches (boundary, generator form, bridge test, precision of the sums) differ from the others' in
a batch or at a server run the kernel that reads the switches, alone one that has them compiled in: the same bits, on
grids whose spacing is no power of two (cell offsets then round)."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem
from test_gpu_serving import drain, server_params, submit

pytestmark = pytest.mark.gpu

PATHS = 700


@pytest.mark.parametrize("precision", [W.PREC_FP32_ACC64, W.PREC_FP32_KAHAN])
def test_mixed_switches_equal_alone(precision):
    import torch

    import paper_1504_00084_gb300 as S
    base = W.c0_small_fp64().replace(precision=precision, substeps=16, paths_per_node=PATHS, nx=50, ny=29, px=3, py=2)
    probs = []
    for per, form, bb, bic, mov in [(0, 0, 1, 1, 0), (0, 1, 1, 1, 1), (0, 0, 0, 0, 0), (0, 1, 0, 1, 0), (1, 0, 1, 1, 0),
                                    (1, 1, 1, 0, 0), (1, 1, 0, 1, 0), (0, 1, 1, 0, 0)]:
        probs.append(base.replace(periodic=per, form=form, bb_test=bb, bicubic=bic, moving_boundary=mov, tau=1.0,
                                  dt=1e-3 if form else 3e-3, seed=len(probs) + 1))
    start = [W.sine_mode_mesh(p, amp=0.02, periodic_mode=bool(p.periodic)) for p in probs]
    want = []
    for prob, (x, y) in zip(probs, start):
        h = gpu_problem(prob, x, y)
        want.append(h.step()[:2])
        h.close()
    hs = [gpu_problem(p, x, y) for p, (x, y) in zip(probs, start)]
    stream = torch.cuda.Stream()
    with S.SddBatch(hs, stream=stream) as b:
        b.step()
        b.stats()
    stream.synchronize()
    for prob, h, (x, y) in zip(probs, hs, want):
        gx, gy = h.mesh()
        h.close()
        assert np.array_equal(gx, x) and np.array_equal(gy, y), prob
    with S.SddServer(server_params(precision, PATHS), torch.cuda.Stream()) as srv:
        ids = [submit(srv, p, x, y) for p, (x, y) in zip(probs, start)]
        drain(srv, len(ids))
        for prob, rid, (x, y) in zip(probs, ids, want):
            r = srv.result(rid)
            assert np.array_equal(r["x"], x) and np.array_equal(r["y"], y), prob
