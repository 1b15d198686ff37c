"""Compensated FP32 sums on both sides of the line at which their tasks are split (8192 paths a node): their distance
from FP64 sums over the same paths, and that a batch and a server group and run a problem's paths as the problem alone
does.  A compensated add rounds the path's value less the shift, the compensated value and (the first few of a
lane) the lost part, each by at most 2^-24 of the value, 2.53e-8 of it in the root mean square: over n paths the mean
is off by at most sqrt(3) 2.53e-8 rms / sqrt(n) as one standard deviation, taken six times."""
import numpy as np
import pytest

import workloads as W
from gpu_helpers import gpu_problem
from test_gpu_serving import drain, server_params, submit

pytestmark = pytest.mark.gpu


def _prob(periodic, paths, **kw):
    return W.c0_small_fp64().replace(precision=W.PREC_FP32_KAHAN, periodic=periodic, form=1, tau=1.0, dt=1e-3,
                                     substeps=16, paths_per_node=paths, **kw)


@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("paths", [8191, 8192])
def test_distance_from_fp64_sums(paths, periodic):
    out = []
    for precision in (W.PREC_FP32_KAHAN, W.PREC_FP32_ACC64):
        h = gpu_problem(_prob(periodic, paths).replace(precision=precision))
        nodes = h.nodes()
        out.append(h.interface_mc()[:2])
        h.close()
    (est, _), (ref, se) = out
    x, y = W.identity_mesh(_prob(periodic, paths))
    at = np.stack([x[nodes[:, 1], nodes[:, 0]], y[nodes[:, 1], nodes[:, 0]]], 1)
    rms = np.sqrt(se ** 2 * paths + (ref - at) ** 2)  # of the values less the shift
    bound = 6 * np.sqrt(3) * 2.53e-8 * rms / np.sqrt(paths) + 4e-16
    assert (np.abs(est - ref) <= bound).all()
    assert (est != ref).any()  # the two do sum in different ways


@pytest.mark.parametrize("precision", [W.PREC_FP32_KAHAN, W.PREC_FP32_ACC64])
def test_batch_and_server_equal_alone(precision):
    import torch

    import paper_1504_00084_gb300 as S
    for paths in (8191, 8192):
        probs = [_prob(per, paths, nx=n, ny=m, px=p, py=2, seed=k + 1).replace(precision=precision)
                 for k, (per, n, m, p) in enumerate([(1, 33, 33, 2), (0, 41, 37, 3), (1, 50, 29, 3)])]
        want = []
        for prob in probs:
            h = gpu_problem(prob)
            want.append(h.step()[:2])
            h.close()
        hs = [gpu_problem(p) for p in probs]
        stream = torch.cuda.Stream()
        with S.SddBatch(hs, stream=stream) as b:
            b.step()
            b.stats()
        stream.synchronize()
        for h, (x, y) in zip(hs, want):
            gx, gy = h.mesh()
            h.close()
            assert np.array_equal(gx, x) and np.array_equal(gy, y)
        with S.SddServer(server_params(precision, paths), torch.cuda.Stream()) as srv:
            ids = [submit(srv, p) for p in probs]
            drain(srv, len(ids))
            for rid, (x, y) in zip(ids, want):
                r = srv.result(rid)
                assert np.array_equal(r["x"], x) and np.array_equal(r["y"], y)
