"""Subdomain solves on chip at extents and monitors far from order 1.  Every quantity of a solve scales exactly with
powers of two, so the mesh and the reported residual have to be the unit problem's bits, scaled: one component may
be scaled without the other, and form 1 does not change with the monitor's size.  Sizes: a few nodes without a coarse
level, one CTA (four warps, sixteen), clusters."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem

pytestmark = pytest.mark.gpu

SIZES = [(4, 5, 1, 1), (33, 33, 2, 2), (66, 66, 1, 1), (130, 131, 1, 1), (202, 180, 1, 1)]


def _step(nx, ny, px, py, form, precision, ex=0, ey=0, ew=0):
    prob = W.c0_small_fp64().replace(nx=nx, ny=ny, px=px, py=py, form=form, precision=precision, dt=1e-3,
                                     tau=1.0 if form else 1e-2, solve_rtol=1e-10, monitor_kind=W.MONITOR_NODAL,
                                     monitor_params=[])
    x, y = W.sine_mode_mesh(prob, amp=0.03)
    om = 1.0 + 8.0 * np.exp(-30.0 * ((x - 0.4) ** 2 + (y - 0.6) ** 2))
    h = gpu_problem(prob.replace(Lx=2.0 ** ex, Ly=2.0 ** ey), np.ldexp(x, ex), np.ldexp(y, ey), omega=np.ldexp(om, ew))
    nodes = h.nodes()
    iface = np.stack([x[nodes[:, 1], nodes[:, 0]] + 0.003, y[nodes[:, 1], nodes[:, 0]] - 0.002], 1)
    gx, gy, status = h.step_from_interface(np.ldexp(iface, [ex, ey]) if len(nodes) else iface)
    st = h.stats()
    h.close()
    assert status == 0 and st["solve_rel_residual"] <= prob.solve_rtol
    return np.ldexp(gx, -ex), np.ldexp(gy, -ey), (st["solve_rel_residual"], st["solve_iters_max"], st["solve_outer_max"])


def _same(a, b):
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[2] == b[2]


@pytest.mark.parametrize("precision", [W.PREC_FP64, W.PREC_FP32_ACC64])
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("size", SIZES)
def test_extents(size, form, precision):
    ref = _step(*size, form, precision)
    for ex, ey in [(-66, -66), (-40, -40), (40, 40), (83, 83), (-66, 83), (300, -300)]:
        _same(_step(*size, form, precision, ex, ey), ref)


@pytest.mark.parametrize("size", SIZES)
def test_monitor_size_fp32(size):
    ref = _step(*size, 1, W.PREC_FP32_ACC64)
    for ew in (-40, 40):
        _same(_step(*size, 1, W.PREC_FP32_ACC64, ew=ew), ref)


@pytest.mark.parametrize("size", SIZES)
def test_monitor_size_fp64(size):
    ref = _step(*size, 1, W.PREC_FP64)
    for ew in (-300, -140, -70, 60, 130, 300):
        _same(_step(*size, 1, W.PREC_FP64, ew=ew), ref)


@pytest.mark.parametrize("form,e", [(0, 8), (1, 8), (1, 18)])
def test_contrast_fp64(form, e):
    """A monitor from 10^-e to 10^e, as far as an FP64 cycle takes the solve to its target (at form 0, the rounding
    of an FP64 residual alone is beyond it from e = 10 on): the solve gets there."""
    prob = W.c0_small_fp64().replace(nx=66, ny=66, px=1, py=1, form=form, precision=W.PREC_FP64, dt=1e-3,
                                     tau=1.0 if form else 1e-2, solve_rtol=1e-8, monitor_kind=W.MONITOR_NODAL,
                                     monitor_params=[])
    x, y = W.identity_mesh(prob)
    h = gpu_problem(prob, x, y, omega=10.0 ** (e * np.sin(2 * np.pi * x) * np.sin(2 * np.pi * y)))
    _, _, status = h.step()
    st = h.stats()
    h.close()
    assert status == 0 and st["solve_rel_residual"] <= prob.solve_rtol, st
