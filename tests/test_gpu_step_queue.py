"""A step queues its Monte Carlo, its solves and the copies of its results before it waits once: the same bits
as the two phases called one after the other, for results that pass through the staging block, larger ones and
device ones; totals equal to sums over the nodes; an invalid monitor leaves the state and the outputs alone."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,px,py,scheme", [
    (33, 33, 2, 2, 0), (3, 3, 1, 1, 0), (181, 180, 2, 2, 0), (201, 201, 2, 1, 0),  # 512 KiB lies between
    (300, 310, 2, 1, 0),                                                           # cluster
    (600, 40, 1, 1, 0),                                                            # from global memory
    (40, 61, 1, 2, 1), (300, 400, 2, 2, 1),
])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_ACC64])
@pytest.mark.parametrize("out", ["host", "device"])
def test_step_is_its_phases(nx, ny, px, py, scheme, precision, out):
    import torch

    import paper_1504_00084_gb300 as S
    prob = W.c0_small_fp64().replace(precision=precision, nx=nx, ny=ny, px=px, py=py, subdomain_scheme=scheme, tau=1.0,
                                     dt=1e-4, substeps=4, paths_per_node=50, monitor_kind=W.MONITOR_NODAL,
                                     monitor_params=[])
    x, y = W.sine_mode_mesh(prob, amp=0.02)
    om = 1.0 + 0.5 * np.sin(3 * x) ** 2
    bad = om.copy()
    bad[ny // 2, nx // 2] = np.nan
    h, ref = gpu_problem(prob, x, y, omega=bad), gpu_problem(prob, x, y, omega=om)
    if out == "host":
        gx, gy = np.full((ny, nx), 7.0), np.full((ny, nx), 7.0)
    else:
        gx, gy = (torch.full((ny, nx), 7.0, dtype=torch.float64, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
    host = (lambda a: a) if out == "host" else (lambda a: a.cpu().numpy())
    with pytest.raises(S.SddError) as e:
        S.sdd_step(h.h, gx, gy)
    assert e.value.status == S.SDD_ERR_INVALID_ARG
    assert (host(gx) == 7.0).all() and (host(gy) == 7.0).all()
    mx, my = h.mesh()
    assert np.array_equal(mx, x) and np.array_equal(my, y)
    h.set_monitor(om)
    S.sdd_step(h.h, gx, gy)
    torch.cuda.synchronize()
    est, se, n, _ = ref.interface_mc()
    rx, ry, _ = ref.subdomain_solve()
    assert np.array_equal(host(gx), rx) and np.array_equal(host(gy), ry)
    mx, my = h.mesh()
    assert np.array_equal(mx, rx) and np.array_equal(my, ry)
    for st in (h.stats(), ref.stats()):
        assert st["paths"] == n.sum() and st["max_se"] == (se.max() if len(se) else 0.0)
    assert h.stats()["path_steps"] == ref.stats()["path_steps"]
    h.close()
    ref.close()
