"""Preparation kernels at the edges of their tiles (32 x 8 nodes) and of the bump monitor's skip rule, against
the oracle.  Tolerances as for the other monitors and paths: omega 1e-14 of its scale (an exponential and a
few roundings), gradients 1e-13 of theirs times the nodes of a side, path values 1e-12 (FP64) / 1e-5 (FP32)."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import compare_node_paths, gpu_problem, oracle_inputs
from oracle import step as ostep
from oracle.monitor import fd_gradient

pytestmark = pytest.mark.gpu

SHAPES = [(31, 7), (32, 8), (33, 9), (34, 10), (65, 17), (8, 64), (300, 140)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("bumps", [
    [9.0, 0.05, 0.3, 0.7, 0.0, 0.2, 0.5, 0.5, 1e-3, 0.02, 0.9, 0.1],  # most terms are skipped
    [1e6, 0.1, 0.5, 0.5, 3.0, 1e-60, 0.5, 0.5],                       # large; one too narrow to see
    [-0.5, 0.2, 0.4, 0.4, 20.0, 0.03, 0.6, 0.6],                      # a negative one: nothing is skipped
], ids=["far", "large", "negative"])
def test_bumps_and_gradient(nx, ny, periodic, bumps):
    prob = W.c3_mix(4)[1].replace(precision=W.PREC_FP64, nx=nx, ny=ny, px=1, py=1, periodic=periodic,
                                  monitor_params=bumps)
    x, y = W.sine_mode_mesh(prob, amp=0.01, periodic_mode=bool(periodic))
    h = gpu_problem(prob, x, y)
    w, wx, we = h.monitor()
    h.close()
    om = ostep.monitor_on_mesh(prob, x, y, prob.t0)
    gx, gy = fd_gradient(om, periodic)
    scale = np.abs(om).max()
    assert np.abs(w - om).max() <= 1e-14 * scale
    gscale = max(np.abs(gx).max(), np.abs(gy).max(), 1.0)
    assert np.abs(wx - gx).max() <= 1e-13 * gscale * nx
    assert np.abs(we - gy).max() <= 1e-13 * gscale * ny


@pytest.mark.parametrize("nx,ny", SHAPES[:6])
@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_ACC64])
def test_packed_records(nx, ny, periodic, precision):
    """Paths of a few substeps from every interface node read the cells around it."""
    prob = W.c0_small_fp64().replace(precision=precision, nx=nx, ny=ny, px=3, py=2, periodic=periodic, tau=1.0,
                                     substeps=4, dt=4e-4)
    x, y = W.sine_mode_mesh(prob, amp=0.02, periodic_mode=bool(periodic))
    h = gpu_problem(prob, x, y)
    om, inp, nodes = oracle_inputs(prob, x, y, prob.t0, 0)
    compare_node_paths(h, inp, nodes, range(0, len(nodes), 3), 40, prob).check()
    h.close()
