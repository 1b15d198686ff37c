"""Forward-Euler subdomains on chip (one CTA, clusters, and a subdomain too large for them) and the moving
boundary's parallel solve, against the oracle in FP64.  Tolerances: the step's interface values are the
oracle's within 1e-10; a forward-Euler substep is a convex combination whose rounding is a few 1e-16, a
boundary solve that of a diagonally dominant system."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem
from oracle import step as ostep
from oracle.boundary import boundary_arrays, boundary_mesh_step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,px,py", [(33, 33, 2, 2), (9, 7, 4, 3), (40, 61, 1, 2), (3, 90, 1, 3), (120, 37, 2, 1),
                                         (66, 66, 1, 1), (200, 150, 1, 1)])
@pytest.mark.parametrize("form", [0, 1])
def test_forward_euler_step_matches_oracle(nx, ny, px, py, form):
    prob = W.c0_small_fp64().replace(nx=nx, ny=ny, px=px, py=py, form=form, tau=1.0, dt=2e-3, substeps=4,
                                     paths_per_node=50, subdomain_scheme=1)
    x, y = W.sine_mode_mesh(prob, amp=0.02)
    h = gpu_problem(prob, x, y)
    gx, gy, status = h.step()
    assert status == 0
    h.close()
    r = ostep.step(prob, x, y, prob.t0, 0)
    assert np.abs(gx - r["x"]).max() <= 1e-10 and np.abs(gy - r["y"]).max() <= 1e-10


@pytest.mark.parametrize("nx,ny", [(3, 3), (4, 5), (33, 66), (130, 70), (4400, 3)])
@pytest.mark.parametrize("form", [0, 1])
def test_moving_boundary_matches_oracle(nx, ny, form):
    prob = W.c0_small_fp64().replace(nx=nx, ny=ny, px=1, py=1, form=form, tau=1.0, dt=1e-3, moving_boundary=1,
                                     monitor_params=[10.0, 8.0, 0.5, 0.2])
    x, y = W.identity_mesh(prob)
    h = gpu_problem(prob, x, y)
    gx, gy, status = h.step()
    assert status == 0
    h.close()
    om = ostep.monitor_on_mesh(prob, x, y, prob.t0)
    bx, by = boundary_arrays(prob, boundary_mesh_step(prob, om, x, y))
    # rounding times the condition of the sides' systems, 1 + 4 r max(omega) / h^2
    tol = max(1e-12, 1e-15 * (1 + 4 * prob.dt / prob.tau * om.max() * (max(nx, ny) - 1) ** 2))
    for sl in (np.s_[0, :], np.s_[-1, :], np.s_[:, 0], np.s_[:, -1]):
        assert np.abs(gx[sl] - bx[sl]).max() <= tol and np.abs(gy[sl] - by[sl]).max() <= tol
