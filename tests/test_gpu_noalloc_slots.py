"""The allocation-free interface Monte Carlo where the slots of its problem's fine tasks do not fit the fixed scratch array
beside a large grid: it runs tasks of twice the size.  The same paths in other groups, so sums of 7000 values of order
1 differ by less than 7000 2^-53 relative; where they fit, bit for bit."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,same", [(370, False), (328, True)])
def test_task_slots_beyond_the_scratch(n, same):
    import torch

    import paper_1504_00084_gb300 as S
    prob = W.c0_small_fp64().replace(precision=W.PREC_FP32_ACC64, nx=n, ny=n, px=3, py=3, periodic=1, form=1, tau=1.0,
                                     dt=1e-3, substeps=100, paths_per_node=7000, monitor_kind=W.MONITOR_NODAL,
                                     monitor_params=[])
    x, y = W.identity_mesh(prob)
    om = 1.0 + 0.5 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    params = S.params_from(prob)
    with S.SddProblem(params, x, y) as h:
        h.set_monitor(om)
        ref, rse, _, _ = h.interface_mc()
    d = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (x, y, om)]
    est = torch.empty(ref.shape, dtype=torch.float64, device="cuda")
    se = torch.empty_like(est)
    assert S.lib.sdd_interface_mc_noalloc(ctypes.byref(params), *[t.data_ptr() for t in d], 0, est.data_ptr(),
                                          se.data_ptr(), torch.cuda.current_stream().cuda_stream) == S.SDD_OK
    torch.cuda.synchronize()
    est, se = est.cpu().numpy(), se.cpu().numpy()
    assert (np.array_equal(est, ref) and np.array_equal(se, rse)) == same
    assert np.abs(est - ref).max() <= 1e-12 and np.abs(se - rse).max() <= 1e-12
