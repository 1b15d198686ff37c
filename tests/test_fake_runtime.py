"""Host side of the library on a CUDA runtime without a GPU (fake_cudart.cpp, preloaded): what a call queues,
in which order it waits and which launches it chooses."""
import ctypes
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    cxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not cxx or not os.path.isdir(cuda):
        pytest.skip("needs g++ and the CUDA headers")
    import __graft_entry__
    __graft_entry__.build()
    lib = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run([cxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", cuda, os.path.join(HERE, "fake_cudart.cpp"),
                    "-o", lib], check=True, timeout=300)

    def run(name, **env):
        r = subprocess.run([sys.executable, os.path.abspath(__file__), lib, name], cwd=ROOT, capture_output=True,
                           text=True, timeout=300, env=dict(os.environ, LD_PRELOAD=lib, PYTHONPATH=ROOT, **env))
        assert r.returncode == 0, (r.stdout + r.stderr)[-4000:]
        return r.stdout
    return run


def problem(**kw):
    import paper_1504_00084_gb300 as S
    import workloads as W
    prob = W.c0_small_fp64().replace(**kw)
    x, y = W.identity_mesh(prob)
    h = S.SddProblem(S.params_from(prob), x, y)
    if prob.monitor_kind != W.MONITOR_NODAL:
        h.set_monitor_analytic(prob.monitor_kind, prob.monitor_params)
    return h


def tune(lib):
    """Every problem its own shape: records that are rewritten differ from those being uploaded."""
    import paper_1504_00084_gb300 as S
    hs = [problem(nx=n, ny=n, seed=n, precision=1) for n in (33, 41, 65)]
    with S.SddBatch(hs, stream=7) as b:
        for sizes in (False, True):
            b.tune_mc(sizes)
            assert lib.fake_races() == 0, "pinned records rewritten before their upload was waited for"


def test_batch_tuning_waits_for_its_uploads(fake):
    fake("tune")


def path_range(lib):
    import paper_1504_00084_gb300 as S
    h = problem()
    before = lib.fake_launches()
    for begin, n in ((1, 2 ** 63 - 1), (2 ** 32, 1), (2 ** 32 - 5, 6), (-1, 2), (0, 0), (2 ** 63 - 1, 1)):
        assert S.lib.sdd_debug_paths(h.h, 0, begin, n, None, None, None) == S.SDD_ERR_INVALID_ARG, (begin, n)
    assert lib.fake_launches() == before
    h.close()


def test_path_ranges_beyond_the_index_are_refused(fake):
    fake("path_range")


def clusters(lib):
    """Solves whose team would be wider than the device's widest cluster go to narrower teams or to global memory."""
    import paper_1504_00084_gb300 as S
    widest = int(os.environ["FAKE_CLUSTER"])
    for kw in (dict(nx=258, ny=258), dict(nx=130, ny=129), dict(nx=120, ny=120, subdomain_scheme=1),
               dict(nx=66, ny=66, subdomain_scheme=1), dict(nx=33, ny=33)):
        for precision in (0, 1):
            before = len(lib.fake_launches())
            with problem(px=1, py=1, precision=precision, **kw) as h:
                try:
                    h.step()
                except S.SddError:  # nothing ran: no solve has reported convergence
                    pass
            made = [line.rsplit(" ", 4) for line in lib.fake_launches()[before:].decode().splitlines()]
            solves = [m for m in made if "chip_kernel" in m[0] or "items_kernel" in m[0] or "fe_kernel" in m[0]]
            assert len(solves) == 1 and int(solves[0][4]) <= widest, (kw, made)
            on_chip = "chip_kernel" in solves[0][0]
            if kw["nx"] == 33 or (widest == 16 and precision == 1):  # in FP64 256 x 256 fits nowhere
                assert on_chip, (kw, made)
            if kw["nx"] == 258 and widest < 16:
                assert not on_chip, (kw, made)


@pytest.mark.parametrize("widest", [1, 2, 4, 8, 16])
def test_teams_fit_the_device(fake, widest):
    fake("clusters", FAKE_CLUSTER=str(widest))


def euler_launches(lib):
    """Forward-Euler subdomains of uneven sizes (some without an interior) that can all run at once are one launch:
    launches of a problem follow each other, each a chain of substeps."""
    import paper_1504_00084_gb300 as S
    for nx, ny, px, py in ((66, 35, 6, 5), (4, 40, 2, 6), (7, 26, 5, 2), (41, 120, 1, 7), (33, 33, 2, 2), (9, 9, 8, 8)):
        before = len(lib.fake_launches())
        with problem(nx=nx, ny=ny, px=px, py=py, subdomain_scheme=1) as h:
            try:
                h.step()
            except S.SddError:  # nothing ran: no solve has reported convergence
                pass
        made = [line for line in lib.fake_launches()[before:].decode().splitlines() if "fe_" in line]
        assert len(made) == 1, ((nx, ny, px, py), made)


def test_uneven_forward_euler_is_one_launch(fake):
    fake("euler_launches")


if __name__ == "__main__":
    LIB = ctypes.CDLL(sys.argv[1])
    LIB.fake_launches.restype = ctypes.c_char_p
    globals()[sys.argv[2]](LIB)
