"""Task sizes of small Monte Carlo rounds (fill_task_paths): a problem whose whole tasks would leave
warps idle runs finer ones.  The same paths are summed in other groups, so FP64 sums stay within
rounding of the oracle's and path counts are equal; a batch, a server-like second problem and the
allocation-free entry group a problem's paths as the problem alone does (bitwise)."""
import ctypes

import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem, oracle_inputs
from oracle import mc

pytestmark = pytest.mark.gpu


def _prob(precision, periodic, form, paths, substeps):
    return W.c0_small_fp64().replace(precision=precision, periodic=periodic, form=form, paths_per_node=paths,
                                     substeps=substeps, tau=1.0 if form else 1e-2, dt=1e-3 if form else 1e-2)


# paths around one lane each, one task, and one more than a task; unequal remainders
@pytest.mark.parametrize("paths", [2, 31, 33, 1000, 2049])
@pytest.mark.parametrize("periodic,form,substeps", [(0, 0, 100), (1, 1, 16), (1, 1, 1), (0, 1, 20)])
def test_split_rounds_match_oracle_fp64(paths, periodic, form, substeps):
    prob = _prob(W.PREC_FP64, periodic, form, paths, substeps)
    x, y = W.identity_mesh(prob)
    om, inp, nodes = oracle_inputs(prob, x, y, prob.t0, 0)
    oest, ose, on, osteps = mc.interface_mc(prob, x, y, om, nodes, 0, np.float64)
    h = gpu_problem(prob)
    est, se, n, _ = h.interface_mc()
    steps = h.stats()["path_steps"]
    h.close()
    assert np.array_equal(n, on) and steps == int(osteps.sum())
    # sums of at most 2049 values of order 1 regrouped: below 2049 * 2^-53 relative
    assert np.abs(est - oest).max() <= 1e-10 and np.abs(se - ose).max() <= 1e-10


@pytest.mark.parametrize("adaptive", [False, True])
def test_split_problem_is_bitwise_itself_in_a_batch(adaptive):
    """Two form-1 FP32 problems of unlike size, fixed N and adaptive (whose later chunks outgrow the
    fine tasks): meshes after a batched step equal those of each problem alone, bit for bit."""
    import torch

    import paper_1504_00084_gb300 as S
    probs = [_prob(W.PREC_FP32_ACC64, 0, 1, 700, 20).replace(nx=n, ny=n, px=p, py=p, seed=k + 1)
             for k, (n, p) in enumerate([(33, 2), (65, 4)])]
    if adaptive:
        probs = [p.replace(se_target=2e-4, max_paths_per_node=1 << 16) for p in probs]
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


def test_noalloc_groups_as_interface_mc():
    import torch

    import paper_1504_00084_gb300 as S
    prob = _prob(W.PREC_FP32_ACC64, 0, 1, 1000, 20).replace(monitor_kind=W.MONITOR_NODAL, monitor_params=[])
    x, y = W.identity_mesh(prob)
    om = 1.0 + x + 0.5 * y
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
    assert np.array_equal(est.cpu().numpy(), ref) and np.array_equal(se.cpu().numpy(), rse)
