"""Moving boundaries in a batch: a side is solved by the method of its own length (parallel up to 4266 nodes,
serial beyond), so that each problem's mesh is bitwise its own alone, whatever the other problems' sides are."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_ACC64])
@pytest.mark.parametrize("shapes", [[(200, 90), (4400, 3), (33, 33)], [(4267, 5), (4266, 5), (7, 4266)], [(9, 300)]])
def test_sides_in_a_batch_equal_alone(shapes, precision):
    import torch

    import paper_1504_00084_gb300 as S
    base = W.c0_small_fp64().replace(px=1, py=1, tau=1.0, dt=1e-5, moving_boundary=1, precision=precision,
                                     monitor_params=[10.0, 8.0, 0.5, 0.2])
    probs = [base.replace(nx=nx, ny=ny, seed=k + 1) for k, (nx, ny) in enumerate(shapes)]
    hs = [gpu_problem(p) for p in probs]
    stream = torch.cuda.Stream()
    with S.SddBatch(hs, stream=stream) as b:
        b.step()
        b.stats()
    stream.synchronize()
    for prob, h in zip(probs, hs):
        gx, gy = h.mesh()
        h.close()
        a = gpu_problem(prob)
        rx, ry, _ = a.step()
        a.close()
        assert np.array_equal(gx, rx) and np.array_equal(gy, ry)
