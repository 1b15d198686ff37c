"""Monitors far from order 1, FP64 paths of form 1 (drift grad omega / omega, unchanged by a scale of omega): a
power-of-two scale changes the estimates by no more than the quotients' last bits, over 500 paths of 20 substeps; and
a monitor whose quotients are infinite gives the oracle's paths."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem
from oracle import mc
from oracle.layout import interface_nodes

pytestmark = pytest.mark.gpu


def _prob():
    return W.c0_small_fp64().replace(form=1, tau=1.0, dt=2e-3, substeps=20, paths_per_node=500,
                                     monitor_kind=W.MONITOR_NODAL, monitor_params=[])


def _estimates(prob, omega):
    h = gpu_problem(prob, omega=np.ascontiguousarray(omega))
    est, se, _, _ = h.interface_mc()
    h.close()
    return est, se


@pytest.mark.parametrize("e", [-900, -130, -126, -124, 122, 124, 125, 126, 127, 128, 900])
def test_scaled_monitor_keeps_estimates(e):
    prob = _prob()
    x, y = W.identity_mesh(prob)
    om = 1.0 + 0.9 * np.sin(3 * np.pi * x) * np.sin(2 * np.pi * y)
    ref, rse = _estimates(prob, om)
    est, se = _estimates(prob, np.ldexp(om, e))
    assert np.abs(est - ref).max() <= 1e-12 and np.abs(se - rse).max() <= 1e-12


def test_infinite_quotients_match_oracle():
    prob = _prob()
    x, y = W.identity_mesh(prob)
    om = np.full_like(x, 1e-30)
    om[10, 10] = 1e300
    est, se = _estimates(prob, om)
    nodes = interface_nodes(prob.nx, prob.ny, prob.px, prob.py, prob.periodic)
    oest, ose, _, _ = mc.interface_mc(prob, x, y, om, nodes, 0, np.float64)
    assert np.isfinite(oest).all()
    assert np.abs(est - oest).max() <= 1e-10 and np.abs(se - ose).max() <= 1e-10
