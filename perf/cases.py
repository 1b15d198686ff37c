"""The calls whose speed is looked after: what users of the mesh generator run, through its public entry points.

Families (the "kind" of a case):
  step     one alternating step, monitor preparation + interface Monte Carlo + subdomain solves
  mc       the interface Monte Carlo alone (callers that solve elsewhere, or split nodes over processes)
  noalloc  the allocation-free interface Monte Carlo on a caller's device buffers
  solve    the subdomain solves alone, from given interface data
  batch    one step of a batch of uneven problems in a CUDA graph
  serve    requests through the continuous-batching server, to their results
"""
import math

import numpy as np
import torch

import paper_1504_00084_gb300 as S

NODAL, GAUSS, FRONT, BUMPS, RINGS = 0, 1, 2, 3, 4
FP64, FP32_ACC64, FP32_KAHAN = 0, 1, 2

DEFAULTS = dict(periodic=0, form=0, precision=FP64, bicubic=1, bb_test=1, substeps=100, solve_max_iter=20000,
                iface_stride=0, L=1.0, tau=1e-2, dt=1e-3, paths=1000, max_paths=0, se_target=0.0, rtol=1e-10,
                scheme=0, moving=0, monitor="gauss", mesh=0.0)


def listed():
    return [
        # The plan's small parity problem, one whole step with host arrays in and out: the smallest step anyone takes.
        dict(name="step_gauss33_fp64", kind="step", nx=33, ny=33, px=2, py=2, dt=1e-2, paths=1000, rtol=1e-12,
             monitor="gauss", path_len=3.9, host=True),
        # The paper's five-ring experiment (Sec. 4.2) at its own sizes: periodic, paper's generator, one substep.
        dict(name="step_rings41_fp64", kind="step", nx=41, ny=41, px=3, py=3, periodic=1, form=1, L=2.0, tau=1.0,
             dt=5e-4, substeps=1, paths=10000, rtol=1e-12, monitor="rings", path_len=1.0, host=True),
        # A ragged grid and split with every option of a mesh coupled to a physical solver: nodal monitor replaced
        # each step, moving boundary, the paper's forward-Euler subdomain steps, FP32 paths.
        dict(name="step_nodal200x141", kind="step", nx=200, ny=141, px=3, py=5, form=1, tau=1.0, dt=5e-4,
             precision=FP32_ACC64, paths=1000, moving=1, scheme=1, monitor="nodal", mesh=0.02, path_len=99.0),
        # The smallest call: a small grid inside somebody else's loop, device buffers only, no allocation.
        dict(name="noalloc65_fp32", kind="noalloc", nx=65, ny=65, px=2, py=2, form=1, tau=1.0, precision=FP32_ACC64,
             substeps=20, paths=1000, monitor="nodal", mesh=0.02, path_len=20.0),
        # The plan's headline configuration: moving front on 257^2 / 4x4, 1e5 compensated FP32 paths per node.
        dict(name="mc_front257_kahan", kind="mc", nx=257, ny=257, px=4, py=4, precision=FP32_KAHAN, paths=100000,
             monitor="front", path_len=6.25),
        # The same grid in the paper's generator form, resolved: long paths, adaptive to a standard error.
        dict(name="mc_front257_adaptive", kind="mc", nx=257, ny=257, px=4, py=4, form=1, tau=1.0,
             precision=FP32_KAHAN, paths=10000, max_paths=1 << 20, se_target=3e-4, monitor="front", path_len=97.5,
             paths_taken=23850),
        # Doubly periodic front, the paper's form, FP64 sums: no exit tests, every path runs all its substeps.
        dict(name="mc_periodic257", kind="mc", nx=257, ny=257, px=4, py=4, periodic=1, form=1, tau=1.0,
             precision=FP32_ACC64, paths=4000, monitor="front", path_len=100.0),
        # The precision sweep's FP64 column: 257^2 sine mode, omega = 1.
        dict(name="mc_sine257_fp64", kind="mc", nx=257, ny=257, px=4, py=4, precision=FP64, paths=500, monitor="one",
             mesh=0.05, path_len=38.0),
        # The 16 subdomain solves of the headline grid from given interface data (63^2 unknowns each).
        dict(name="solve_front257_4x4", kind="solve", nx=257, ny=257, px=4, py=4, precision=FP32_ACC64,
             monitor="front", mesh=0.01),
        # Near the size limit: 4097^2 nodes, 256 subdomains of 255^2 unknowns.
        dict(name="solve_bumps4097_16x16", kind="solve", nx=4097, ny=4097, px=16, py=16, precision=FP32_ACC64,
             monitor="bumps", mesh=0.01),
        # Sixteen of the uneven bump problems stepped together in one CUDA graph.
        dict(name="batch_mix16", kind="batch", count=16, shapes=12345, nmax=513, precision=FP32_ACC64, paths=2000,
             monitor="bumps", path_len=15.6),
        # Requests of the same shapes arriving together at a server with a service level.
        dict(name="serve_mix8", kind="serve", count=8, shapes=777, nmax=257, precision=FP32_ACC64, paths=2000,
             max_paths=1 << 20, se_target=5e-3, paths_taken=9500, monitor="bumps", path_len=15.6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step64", "rings", "nodal", "noalloc", "front", "adaptive", "periodic", "sine", "solve",
                       "solve", "batch", "serve"])
    if kind == "step64":
        n = _log_int(rng, 17, 129)
        return dict(kind="step", nx=n, ny=_log_int(rng, 17, 129), px=rng.randint(1, 4), py=rng.randint(2, 4), dt=1e-2,
                    paths=_log_int(rng, 200, 2000), rtol=1e-12, monitor="gauss", path_len=3.9, host=True,
                    form=0, iface_stride=rng.choice([0, 0, 3]))
    if kind == "rings":
        n = rng.choice([41, 61, 81])
        return dict(kind="step", nx=n, ny=n, px=rng.randint(2, 4), py=rng.randint(2, 4), periodic=1, form=1, L=2.0,
                    tau=1.0, dt=5e-4, substeps=rng.choice([1, 16]), paths=_log_int(rng, 1000, 10000), rtol=1e-12,
                    monitor="rings", path_len=8.0, host=True)
    if kind == "nodal":
        return dict(kind="step", nx=rng.randint(40, 260), ny=rng.randint(40, 260), px=rng.randint(2, 6),
                    py=rng.randint(2, 6), form=1, tau=1.0, dt=5e-4, precision=rng.choice([FP32_ACC64, FP32_KAHAN]),
                    paths=_log_int(rng, 300, 3000), moving=rng.randint(0, 1), scheme=rng.randint(0, 1),
                    bicubic=rng.choice([1, 1, 0]), bb_test=rng.choice([1, 1, 0]), monitor="nodal", mesh=0.02,
                    path_len=99.0)
    if kind == "noalloc":
        p = rng.choice([2, 3, 4])
        return dict(kind="noalloc", nx=p * rng.randint(8, 40) + 1, ny=p * rng.randint(8, 40) + 1, px=p, py=p, form=1,
                    tau=1.0, precision=rng.choice([FP64, FP32_ACC64, FP32_KAHAN]), substeps=rng.randint(5, 100),
                    paths=_log_int(rng, 200, 20000), monitor="nodal", mesh=0.02, path_len=50.0)
    if kind == "front":
        n = _log_int(rng, 129, 400)
        return dict(kind="mc", nx=n, ny=_log_int(rng, 129, 400), px=rng.randint(2, 6), py=rng.randint(2, 6),
                    precision=rng.choice([FP32_ACC64, FP32_KAHAN]), paths=_log_int(rng, 5000, 100000),
                    monitor="front", path_len=6.25)
    if kind == "adaptive":
        n = _log_int(rng, 129, 257)
        return dict(kind="mc", nx=n, ny=n, px=rng.randint(2, 4), py=rng.randint(2, 4), form=1, tau=1.0,
                    precision=rng.choice([FP32_ACC64, FP32_KAHAN]), paths=_log_int(rng, 2000, 10000),
                    max_paths=1 << 20, se_target=rng.choice([3e-4, 5e-4, 1e-3]), monitor="front", path_len=97.5,
                    paths_taken=12000)
    if kind == "periodic":
        return dict(kind="mc", nx=_log_int(rng, 65, 257), ny=_log_int(rng, 65, 257), px=rng.randint(2, 4),
                    py=rng.randint(2, 4), periodic=1, form=1, tau=1.0, precision=rng.choice([FP32_ACC64, FP32_KAHAN]),
                    paths=_log_int(rng, 500, 4000), monitor="front", path_len=100.0)
    if kind == "sine":
        return dict(kind="mc", nx=_log_int(rng, 65, 257), ny=_log_int(rng, 65, 257), px=rng.randint(2, 4),
                    py=rng.randint(2, 4), precision=FP64, paths=_log_int(rng, 100, 500), monitor="one", mesh=0.05,
                    path_len=38.0)
    if kind == "solve":
        n = _log_int(rng, 33, 1500)
        p = max(2, n // rng.randint(30, 270))
        return dict(kind="solve", nx=n, ny=_log_int(rng, 33, 1500), px=p, py=rng.randint(2, 6), form=rng.randint(0, 1),
                    precision=rng.choice([FP32_ACC64, FP32_ACC64, FP64]), monitor=rng.choice(["gauss", "bumps"]),
                    mesh=0.01)
    c = dict(kind=kind, count=rng.randint(3, 8), shapes=rng.randint(1, 1 << 20), nmax=rng.choice([129, 257]),
             precision=rng.choice([FP32_ACC64, FP32_KAHAN]), paths=_log_int(rng, 500, 2000), monitor="bumps",
             path_len=15.6)
    if kind == "serve":
        c.update(max_paths=1 << 20, se_target=rng.choice([5e-3, 1e-2]), paths_taken=5000)
    return c


# ---------------------------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------------------------

def _full(case):
    return {**DEFAULTS, **case}


def _params(c, seed, **over):
    p = S.SddParams()
    for k in ("nx", "ny", "px", "py", "periodic", "form", "precision", "bicubic", "bb_test", "substeps",
              "solve_max_iter", "iface_stride", "tau", "dt", "se_target"):
        setattr(p, k, c[k])
    p.Lx = p.Ly = c["L"]
    p.seed = seed + 1
    p.paths_per_node = c["paths"]
    p.max_paths_per_node = c["max_paths"] or c["paths"]
    p.solve_rtol = c["rtol"]
    p.subdomain_scheme = c["scheme"]
    p.moving_boundary = c["moving"]
    for k, v in over.items():
        setattr(p, k, v)
    return p


def _monitor(c, rng):
    """(kind, parameters) of an analytic monitor; centres and strengths move a little with the seed."""
    j = lambda: float(rng.uniform(-0.02, 0.02))  # noqa: E731
    if c["monitor"] == "gauss":
        return GAUSS, [10.0 + 20 * j(), 50.0, 0.5 + j(), 0.5 + j()]
    if c["monitor"] == "front":
        return FRONT, [50.0, 50.0, 0.25 + 0.2 * j(), 0.1, 0.5 + 0.2 * j(), 0.5 + 0.2 * j()]
    if c["monitor"] == "rings":
        o = [j() for _ in range(2)]
        return RINGS, [0.2, 30.0, 0.125, 1.0 + o[0], 1.0 + o[1], 0.5, 0.5, 0.5, 1.5, 1.5, 0.5, 1.5, 1.5]
    if c["monitor"] == "bumps":
        q = []
        for _ in range(3):
            q += [float(rng.uniform(1.0, 20.0)), float(rng.uniform(0.02, 0.1)), float(rng.uniform(0.1, 0.9)),
                  float(rng.uniform(0.1, 0.9))]
        return BUMPS, q
    return BUMPS, []  # "one": omega = 1


def _mesh(c, rng):
    """Identity plus sine modes of total amplitude "mesh" (zero at the boundary): a mesh some steps into a run."""
    xi = np.arange(c["nx"], dtype=np.float64) / (c["nx"] - 1)
    eta = np.arange(c["ny"], dtype=np.float64) / (c["ny"] - 1)
    x = np.broadcast_to(c["L"] * xi[None, :], (c["ny"], c["nx"])).copy()
    y = np.broadcast_to(c["L"] * eta[:, None], (c["ny"], c["nx"])).copy()
    if c["mesh"]:
        k = 2 if c["periodic"] else 1
        for f in (x, y):
            a, b = c["mesh"] * rng.uniform(0.5, 1.0), 0.2 * c["mesh"] * rng.uniform(-1, 1)
            for amp, m in ((a, k), (b, 2 * k)):
                su, sv = np.sin(m * np.pi * eta), np.sin(m * np.pi * xi)
                su[-1] = sv[-1] = 0.0
                f += amp * c["L"] * np.outer(su, sv)
    return x, y


def _nodal(c, x, y, rng):
    cx, cy = c["L"] * (0.5 + 0.05 * rng.uniform(-1, 1)), c["L"] * (0.5 + 0.05 * rng.uniform(-1, 1))
    w = 1.0 + 4.0 * np.exp(-30.0 * ((x - cx) ** 2 + (y - cy) ** 2) / c["L"] ** 2)
    if c["periodic"]:
        w[:, -1], w[-1, :] = w[:, 0], w[0, :]
    return w


def _iface(c, nodes, rng):
    """Interface data of a solve: the nodes' own places moved along smooth modes."""
    xi, eta = nodes[:, 0] / (c["nx"] - 1.0), nodes[:, 1] / (c["ny"] - 1.0)
    a = 0.01 * rng.uniform(0.5, 1.5, size=2)
    s = np.sin(np.pi * xi) * np.sin(2 * np.pi * eta) if not c["periodic"] else np.sin(2 * np.pi * xi) * np.sin(2 * np.pi * eta)
    return c["L"] * np.stack([xi + a[0] * s, eta - a[1] * s], axis=1)


def _shapes(c):
    rng = np.random.default_rng(c["shapes"])
    got = []
    for _ in range(c["count"]):
        n = int(rng.choice([v for v in (65, 100, 129, 200, 257, 513) if v <= c["nmax"]]))
        p = int(rng.choice([2, 4, 8] if n > 65 else [2, 4]))
        got.append((n, p))
    return got


def prepare(case, seed):
    c, rng = _full(case), np.random.default_rng(seed)
    st = {"c": c}
    if c["kind"] in ("batch", "serve"):
        st["stream"] = torch.cuda.Stream()
        made = []
        for k, (n, p) in enumerate(_shapes(c)):
            ck = {**c, "nx": n, "ny": n, "px": p, "py": p}
            made.append((_params(ck, seed + 1000 * k), *_mesh(ck, rng), *_monitor(ck, rng)))
        if c["kind"] == "serve":
            q = S.SddServerParams()
            q.precision, q.max_resident, q.max_nodes, q.mem_budget_bytes = c["precision"], 64, 40000, 0
            q.se_target, q.paths_per_node, q.max_paths_per_node = c["se_target"], c["paths"], c["max_paths"]
            q.round_paths = 0
            st["server"], st["requests"] = S.SddServer(q, st["stream"]), made
            return st
        st["problems"] = []
        for prm, x, y, kind, q in made:
            h = S.SddProblem(prm, x, y, stream=st["stream"])
            h.set_monitor_analytic(kind, q)
            st["problems"].append(h)
        st["batch"] = S.SddBatch(st["problems"], stream=st["stream"], use_graph=True)
        st["out"] = [torch.empty(2, h.ny, h.nx, dtype=torch.float64, device="cuda") for h in st["problems"]]
        torch.cuda.synchronize()
        return st
    x, y = _mesh(c, rng)
    prm = _params(c, seed)
    st["params"] = prm
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    new = lambda *s: torch.empty(*s, dtype=torch.float64, device="cuda")  # noqa: E731
    if c["kind"] == "noalloc":
        st["in"] = dev(x), dev(y), dev(_nodal(c, x, y, rng))
        M = len(S.sdd_interface_layout(c["nx"], c["ny"], c["px"], c["py"], c["periodic"]))
        st["out"] = new(M, 2), new(M, 2)
        torch.cuda.synchronize()
        return st
    h = S.SddProblem(prm, x, y, stream=torch.cuda.current_stream())
    st["h"] = h
    if c["monitor"] == "nodal":
        st["omega"] = dev(_nodal(c, x, y, rng))
        h.set_monitor(st["omega"])
    else:
        h.set_monitor_analytic(*_monitor(c, rng))
    if c["kind"] == "mc":
        st["out"] = new(h.M, 2), new(h.M, 2), torch.empty(h.M, dtype=torch.int64, device="cuda")
    elif c["kind"] == "solve":
        st["iface"] = dev(_iface(c, h.nodes(), rng))
        st["out"] = new(h.ny, h.nx), new(h.ny, h.nx)
    elif not c.get("host"):
        st["out"] = new(h.ny, h.nx), new(h.ny, h.nx)
    torch.cuda.synchronize()
    return st


def run(st):
    c = st["c"]
    if c["kind"] == "noalloc":
        x, y, w = st["in"]
        est, se = st["out"]
        s = S.lib.sdd_interface_mc_noalloc(S.ctypes.byref(st["params"]), x.data_ptr(), y.data_ptr(), w.data_ptr(), 0,
                                           est.data_ptr(), se.data_ptr(), torch.cuda.current_stream().cuda_stream)
        if s != S.SDD_OK:
            raise RuntimeError("sdd_interface_mc_noalloc: status %d" % s)
        return {"est": est, "se": se}
    if c["kind"] == "mc":
        est, se, n = st["out"]
        S.sdd_interface_mc(st["h"].h, est, se, n)
        return {"est": est, "se": se, "paths": n}
    if c["kind"] == "solve":
        x, y = st["out"]
        S.sdd_subdomain_solve(st["h"].h, st["iface"], x, y)
        return {"x": x, "y": y}
    if c["kind"] == "step":
        if c.get("host"):
            x, y, _ = st["h"].step()
            return {"x": x, "y": y}
        x, y = st["out"]
        S.sdd_set_monitor(st["h"].h, st["omega"])
        S.sdd_step(st["h"].h, x, y)
        return {"x": x, "y": y}
    if c["kind"] == "batch":
        st["batch"].step()
        for h, o in zip(st["problems"], st["out"]):
            S.sdd_get_mesh(h.h, o[0], o[1])
        return {"mesh": st["out"]}
    server, ids, done = st["server"], [], {}
    for prm, x, y, kind, q in st["requests"]:
        ids.append(server.submit(prm, x, y, kind, q))
    while len(done) < len(ids):
        server.progress()
        for rid in server.poll():
            done[rid] = server.result(rid)
    return {"results": [{k: done[rid][k] for k in ("x", "y", "est", "se")} for rid in ids]}


def _interface_count(c):
    nx, ny, px, py = c["nx"], c["ny"], c["px"], c["py"]
    if c["periodic"]:
        return px * (ny - 1) + py * (nx - 1) - px * py
    return (px - 1) * (ny - 2) + (py - 1) * (nx - 2) - (px - 1) * (py - 1)


def work(case):
    """Bytes: the mesh and monitor in, the mesh or estimates out.  Operations: 158 (121 periodic) per path substep;
    a solve's matrix is applied and its smoother run a few times at the least (40 operations per unknown)."""
    c = _full(case)
    if c["kind"] in ("batch", "serve"):
        parts = [{**c, "nx": n, "ny": n, "px": p, "py": p} for n, p in _shapes(c)]
    else:
        parts = [c]
    nbytes = flops = 0.0
    for q in parts:
        N, M = q["nx"] * q["ny"], _interface_count(q)
        nbytes += 16.0 * N + (8.0 * N if q["monitor"] == "nodal" else 0.0)
        if q["kind"] != "solve":
            flops += M * q.get("paths_taken", q["paths"]) * q["path_len"] * (121.0 if q["periodic"] else 158.0)
        if q["kind"] in ("mc", "noalloc", "serve"):
            nbytes += 32.0 * M
        if q["kind"] not in ("mc", "noalloc"):
            nbytes += 16.0 * N
            flops += 40.0 * N
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------
# The same results in 64 bits, from the method's definition in plain torch.
# ---------------------------------------------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, key):
    m = 0xFFFFFFFF
    k0, k1 = key & m, (key >> 32) & m
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # 64-bit products; int64 wraps, the bits are those of uint64
        c0, c1, c2, c3 = ((b >> 32) & m) ^ c1 ^ k0, b & m, ((a >> 32) & m) ^ c3 ^ k1, a & m
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2


def _omega(c, kind, q, x, y, t=0.0):
    im = (lambda d: d - c["L"] * torch.floor(d / c["L"] + 0.5)) if c["periodic"] else (lambda d: d)
    if kind == GAUSS:
        return torch.sqrt(1 + q[0] * torch.exp(-q[1] * (im(x - q[2]) ** 2 + im(y - q[3]) ** 2)))
    if kind == FRONT:
        r = torch.sqrt(im(x - q[4]) ** 2 + im(y - q[5]) ** 2)
        u = torch.tanh(q[1] * (r - q[2] - q[3] * t))
        return torch.sqrt(1 + q[0] * (q[1] * (1 - u * u)) ** 2)
    if kind == RINGS:
        gx, gy = torch.zeros_like(x), torch.zeros_like(x)
        for b in range(3, len(q), 2):
            dx, dy = im(x - q[b]), im(y - q[b + 1])
            f = 2 * q[1] * (1 - torch.tanh(q[1] * (dx * dx + dy * dy - q[2])) ** 2)
            gx, gy = gx + f * dx, gy + f * dy
        return torch.sqrt(1 + q[0] * (gx * gx + gy * gy))
    w = torch.ones_like(x)
    for b in range(0, len(q), 4):
        w = w + q[b] * torch.exp(-(im(x - q[b + 2]) ** 2 + im(y - q[b + 3]) ** 2) / q[b + 1] ** 2)
    return w


def _gradient(f, dim, periodic):
    f = f.movedim(dim, 0)
    n, g = f.shape[0], torch.empty_like(f)
    if periodic:
        u = f[:-1]
        g[:-1] = torch.roll(u, -1, 0) - torch.roll(u, 1, 0)
        g[-1] = g[0]
    else:
        g[1:-1] = f[2:] - f[:-2]
        g[0] = -3 * f[0] + 4 * f[1] - f[2]
        g[-1] = 3 * f[-1] - 4 * f[-2] + f[-3]
    return (0.5 * (n - 1) * g).movedim(0, dim)


def _pad(f, periodic):
    """One more node on each side: wrapped, or Keys' extrapolation 3 f0 - 3 f1 + f2."""
    for _ in range(2):
        if periodic:
            f = torch.cat([f[-2:-1], f, f[1:2]])
        else:
            f = torch.cat([(3 * f[0] - 3 * f[1] + f[2])[None], f, (3 * f[-1] - 3 * f[-2] + f[-3])[None]])
        f = f.transpose(0, 1)
    return f.contiguous()


def _keys(t):
    a = [1 + t, t, 1 - t, 2 - t]
    near = lambda s: (1.5 * s - 2.5) * s * s + 1  # noqa: E731
    far = lambda s: ((-0.5 * s + 2.5) * s - 4) * s + 2  # noqa: E731
    return [far(a[0]), near(a[1]), near(a[2]), far(a[3])]


def _cell(n, s, periodic):
    u = s * (n - 1)
    f = torch.floor(u)
    if periodic:
        return torch.remainder(f, n - 1).long(), u - f
    f = f.clamp(0, n - 2)
    return f.long(), u - f


def _paths(c, key, fields, padded, m, ij, p):
    """End values (x, y) of paths p of nodes m, from the counter-based draws."""
    nx, ny, per, L = c["nx"], c["ny"], c["periodic"], c["L"]
    cb = c["dt"] / c["substeps"] / c["tau"]
    vx, vy = torch.empty(p.shape, dtype=torch.float64, device=p.device), None
    vy = torch.empty_like(vx)
    at = torch.arange(p.numel(), device=p.device)
    X, Y = ij[:, 0].double() / (nx - 1), ij[:, 1].double() / (ny - 1)
    for k in range(c["substeps"]):
        i, fx = _cell(nx, X, per)
        j, fy = _cell(ny, Y, per)
        b = j * nx + i
        w = [(1 - fx) * (1 - fy) * f[b] + fx * (1 - fy) * f[b + 1] + (1 - fx) * fy * f[b + nx] + fx * fy * f[b + nx + 1]
             for f in fields]
        r = _philox(torch.full_like(p, k), p, m, torch.zeros_like(p), key)
        if c["precision"] == FP64:
            u1, u2, u3 = [(v.double() + 0.5) * 2.0 ** -32 for v in r]
        else:
            u1, u2, u3 = [((v >> 9).double() + 0.5) * 2.0 ** -23 for v in r]
        q = w[0] * cb if c["form"] == 0 else torch.full_like(X, cb)
        d = cb if c["form"] == 0 else cb / w[0]
        s = torch.sqrt(2 * q) * torch.sqrt(-2 * torch.log(u1))
        xn, yn = X + w[1] * d + s * torch.cos(2 * math.pi * u2), Y + w[2] * d + s * torch.sin(2 * math.pi * u2)
        if per:
            X, Y = xn, yn
            continue
        over = torch.stack([-xn, xn - 1, -yn, yn - 1])
        side = over.argmax(0)
        out = over.max(0).values > 0
        if c["bb_test"]:
            pr = torch.stack([torch.exp(-X * xn / q), torch.exp(-(1 - X) * (1 - xn) / q), torch.exp(-Y * yn / q),
                              torch.exp(-(1 - Y) * (1 - yn) / q)])
            hit = ~out & (u3 > (1 - pr).prod(0))
            side = torch.where(hit, pr.argmax(0), side)
            out = out | hit
        if bool(out.any()):
            xe, ye, so = xn[out].clamp(0, 1), yn[out].clamp(0, 1), side[out]
            xe = torch.where(so == 0, torch.zeros_like(xe), torch.where(so == 1, torch.ones_like(xe), xe))
            ye = torch.where(so == 2, torch.zeros_like(ye), torch.where(so == 3, torch.ones_like(ye), ye))
            vx[at[out]], vy[at[out]] = L * xe, L * ye
            on = ~out
            at, X, Y, p, m = at[on], xn[on], yn[on], p[on], m[on]
        else:
            X, Y = xn, yn
        if not at.numel():
            return vx, vy
    i, fx = _cell(nx, X, per)
    j, fy = _cell(ny, Y, per)
    for v, f, base in ((vx, padded[0], L * X), (vy, padded[1], L * Y)):
        g = f.reshape(-1)
        if c["bicubic"]:
            kx, ky, tot = _keys(fx), _keys(fy), 0.0
            for b in range(4):
                tot = tot + ky[b] * sum(kx[a] * g[(j + b) * (nx + 2) + i + a] for a in range(4))
        else:
            o = (j + 1) * (nx + 2) + i + 1
            tot = ((1 - fx) * (1 - fy) * g[o] + fx * (1 - fy) * g[o + 1] + (1 - fx) * fy * g[o + nx + 2] +
                   fx * fy * g[o + nx + 3])
        v[at] = base + tot
    return vx, vy


def _estimates(c, key, om, x, y, nodes):
    per, N = c["periodic"], c["paths"]
    fields = [om.reshape(-1), _gradient(om, 1, per).reshape(-1), _gradient(om, 0, per).reshape(-1)]
    ident = [c["L"] * torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1) for n in (c["nx"], c["ny"])]
    padded = [_pad(x - ident[0][None, :], per), _pad(y - ident[1][:, None], per)]
    M, step = len(nodes), max(1, 8_000_000 // N)
    est, se = torch.empty(M, 2, dtype=torch.float64, device="cuda"), torch.empty(M, 2, dtype=torch.float64, device="cuda")
    for a in range(0, M, step):
        m = torch.arange(a, min(M, a + step), device="cuda")
        p = torch.arange(N, device="cuda").repeat(len(m))
        mm = m.repeat_interleave(N)
        for k, v in enumerate(_paths(c, key, fields, padded, mm, nodes[mm], p)):
            v = v.reshape(len(m), N)
            est[m, k], se[m, k] = v.mean(1), torch.sqrt(v.var(1) / N)
    return est, se


def _solved(c, om, x, y, nodes, est):
    """The backward-Euler subdomain systems, all at once, by conjugate gradients with FP64 restarts."""
    nx, ny, L, r = c["nx"], c["ny"], c["L"], c["dt"] / c["tau"]
    free = torch.ones(ny, nx, dtype=torch.bool, device="cuda")
    for I in range(c["px"] + 1):
        free[:, I * (nx - 1) // c["px"]] = False
    for J in range(c["py"] + 1):
        free[J * (ny - 1) // c["py"], :] = False
    ce, cn = r * 0.5 * (om[:, 1:] + om[:, :-1]) * (nx - 1) ** 2, r * 0.5 * (om[1:] + om[:-1]) * (ny - 1) ** 2
    d = torch.ones_like(om) if c["form"] == 0 else om
    fm = free.double()

    def apply(v):
        e, n = ce * (v[..., :, 1:] - v[..., :, :-1]), cn * (v[..., 1:, :] - v[..., :-1, :])
        out = d * v
        out[..., :, :-1] -= e
        out[..., :, 1:] += e
        out[..., :-1, :] -= n
        out[..., 1:, :] += n
        return out * fm

    old = torch.stack([x, y])
    ident = torch.stack([(L * torch.arange(nx, dtype=torch.float64, device="cuda") / (nx - 1))[None, :].expand(ny, nx),
                         (L * torch.arange(ny, dtype=torch.float64, device="cuda") / (ny - 1))[:, None].expand(ny, nx)])
    v = torch.where(free, old, ident)
    i, j = nodes[:, 0], nodes[:, 1]
    v[:, j, i] = est.T
    if c["periodic"]:
        v[:, :, -1] = v[:, :, 0] + torch.tensor([L, 0.0], device="cuda", dtype=torch.float64)[:, None]
        v[:, -1, :] = v[:, 0, :] + torch.tensor([0.0, L], device="cuda", dtype=torch.float64)[:, None]
    diag = d.clone()
    diag[:, :-1] += ce
    diag[:, 1:] += ce
    diag[:-1] += cn
    diag[1:] += cn
    for _ in range(3):
        res = (d * old - apply(v)) * fm
        e, z = torch.zeros_like(v), res / diag
        p, rz = z.clone(), (res * z).sum((1, 2))
        first = rz.clone()
        for _ in range(6000):
            q = apply(p)
            a = (rz / (p * q).sum((1, 2)).clamp_min(1e-300))[:, None, None]
            e += a * p
            res -= a * q
            z = res / diag
            new = (res * z).sum((1, 2))
            p = z + (new / rz.clamp_min(1e-300))[:, None, None] * p
            rz = new
            if bool((rz <= 1e-18 * first).all()):
                break
        v += e
    return v[0], v[1]


def _nodes(c):
    """Interface nodes (i, j): vertical lines by i, then the horizontal lines' nodes that are not on those."""
    lo, hi = (0, -1) if c["periodic"] else (1, -1)
    vl = [I * (c["nx"] - 1) // c["px"] for I in range(lo, c["px"])]
    hl = [J * (c["ny"] - 1) // c["py"] for J in range(lo, c["py"])]
    got = [(i, j) for i in vl for j in range(lo, c["ny"] + hi)]
    got += [(i, j) for j in hl for i in range(lo, c["nx"] + hi) if i not in vl]
    return np.array(got, dtype=np.int64).reshape(-1, 2)


def exact(case, seed):
    c, rng = _full(case), np.random.default_rng(seed)
    # Not written out in plain form: path counts that depend on the results, the boundary's own motion and the
    # explicit subdomain steps, sampled interfaces, many problems at once.
    if c["kind"] in ("batch", "serve") or c["se_target"] or c["moving"] or c["scheme"] or c["iface_stride"] > 1:
        return None
    x, y = _mesh(c, rng)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    gx, gy = dev(x), dev(y)
    if c["monitor"] == "nodal":
        om = dev(_nodal(c, x, y, rng))
    else:
        kind, q = _monitor(c, rng)
        om = _omega(c, kind, q, gx, gy)
    if c["periodic"]:
        om[:, -1] = om[:, 0]
        om[-1, :] = om[0, :]
    ij = _nodes(c)
    nodes = dev(ij)
    if c["kind"] == "solve":
        sx, sy = _solved(c, om, gx, gy, nodes, dev(_iface(c, ij, rng)))
        return {"x": sx, "y": sy}
    est, se = _estimates(c, seed + 1, om, gx, gy, nodes)
    if c["kind"] == "noalloc":
        return {"est": est, "se": se}
    if c["kind"] == "mc":
        return {"est": est, "se": se, "paths": None}
    sx, sy = _solved(c, om, gx, gy, nodes, est)
    return {"x": sx, "y": sy}
