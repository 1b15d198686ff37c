"""Subdomain solves held on chip (sdd_chip.cuh) at the sizes where the team changes: one interior node,
the last size of one CTA and the first of a cluster, clusters of 4, 8 and 16, rows wider than 64
(several warps to a row) and than 128, odd and even sizes, long and narrow ones, the first size that
goes back to global memory.  One Dirichlet subdomain against the oracle's direct solve, within the
solver bound of the parity tests; and, split unevenly, in a batch, bit for bit as alone."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem, mesh_tolerance
from oracle import step as ostep
from oracle.solve import single_domain_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_ACC64])
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("ni,nj", [(1, 1), (2, 3), (1, 40), (3, 3), (16, 15), (31, 33), (64, 64), (65, 64), (66, 28),
                                   (28, 66), (100, 99), (128, 129), (200, 90), (256, 256), (257, 40), (40, 257)])
def test_team_sizes_match_oracle(ni, nj, form, precision):
    prob = W.c0_small_fp64().replace(nx=ni + 2, ny=nj + 2, px=1, py=1, precision=precision, form=form,
                                     tau=1.0 if form else 1e-2, dt=1e-3, solve_rtol=1e-11)
    x, y = W.sine_mode_mesh(prob, amp=0.03)
    h = gpu_problem(prob, x, y)
    gx, gy, status = h.step()
    assert status == 0 and h.stats()["solve_rel_residual"] <= prob.solve_rtol
    h.close()
    om = ostep.monitor_on_mesh(prob, x, y, prob.t0)
    ox, oy = single_domain_step(om, x, y, prob.dt, prob.tau, prob.form)
    bx, by = ostep.scatter(prob, np.zeros((0, 2), np.int32), np.zeros((0, 2)))
    tol = mesh_tolerance(prob, om, bx, by, x, y, 0.0)
    assert np.abs(gx - ox).max() <= tol and np.abs(gy - oy).max() <= tol


def test_uneven_teams_in_a_batch_equal_alone():
    """Splits whose parts fall into several teams (and an empty interior), FP32: the meshes of a batched
    step are bitwise those of each problem alone."""
    import torch

    import paper_1504_00084_gb300 as S
    base = W.c0_small_fp64().replace(precision=W.PREC_FP32_ACC64, paths_per_node=64, substeps=4, dt=1e-3)
    probs = [base.replace(nx=n, ny=m, px=p, py=q, seed=k + 1)
             for k, (n, m, p, q) in enumerate([(131, 130, 2, 2), (200, 67, 3, 1), (9, 9, 6, 2), (260, 300, 2, 1)])]
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
