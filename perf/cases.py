"""The work that a user of the library has it do, as timed cases through its public entry points.

The kinds of case:
  advance  one simulation resident on the GPU: advance it by `steps` and read its three fields into host
           arrays (a snapshot, or the end of a run).  `restart`: the fields are first loaded from host arrays
           (a new shot or a restart); without it the simulation goes on from the pass before.  `layers`: absorbing
           layers along the walls.  The nodal scheme grows at its boundary by a few per cent a step, so its runs
           restart or carry layers; the staggered scheme is neutral.
  batch    many simulations of both schemes and uneven sizes advanced together, then read.
  serve    requests submitted to the serving loop, from submission to the host copies of their results: creation,
           source, steps, read-back.
  static   one step between the caller's own device buffers, without allocations.
  iterate  the paper's fixed-point stage solver on host arrays, for comparison with the exact solves.

Grids, media and time steps are the ones that the tests and the benchmark use: the unit square's 100 cells, 1001 x 1001
and 4096 x 4096 seismic grids, batches of 128-1024 cells a side, requests of 64 cells a side and more, 8192-cell lines.
Fields are held in single precision unless `f64` (the convergence studies run in double precision).
"""
import math

import numpy as np
import torch

from paper_2006_07583_gb300 import adi

CFD, MFD = adi.ADI_CFD, adi.ADI_MFD


def listed():
    return [
        # the smallest call: one step between device buffers, for callers that may not allocate
        {"name": "static_cfd_64", "kind": "static", "method": CFD, "nx": 64, "ny": 64, "f64": False},
        # the unit-square problem's grid, a few steps at a time: launches and latency count
        {"name": "snapshot_mfd_100", "kind": "advance", "method": MFD, "nx": 100, "ny": 100, "steps": 25, "f64": False,
         "restart": False, "layers": 0},
        # a convergence study's rung: double precision, restarted from an exact solution's fields
        {"name": "ladder_cfd_512_f64", "kind": "advance", "method": CFD, "nx": 512, "ny": 512, "steps": 8, "f64": True,
         "restart": True, "layers": 0},
        # the reference run in double precision that a single-precision result is compared with
        {"name": "snapshot_mfd_1001_f64", "kind": "advance", "method": MFD, "nx": 1001, "ny": 1001, "steps": 20, "f64": True,
         "restart": False, "layers": 0},
        # a section of a seismic survey, sides that are no round numbers
        {"name": "shot_cfd_1203x777", "kind": "advance", "method": CFD, "nx": 1203, "ny": 777, "steps": 16, "f64": False,
         "restart": True, "layers": 0},
        # a seismic run's snapshots at the usual size
        {"name": "snapshot_mfd_1001", "kind": "advance", "method": MFD, "nx": 1001, "ny": 1001, "steps": 40, "f64": False,
         "restart": False, "layers": 0},
        # the same with absorbing layers, as an unbounded medium needs them
        {"name": "layers_cfd_640", "kind": "advance", "method": CFD, "nx": 640, "ny": 640, "steps": 20, "f64": False,
         "restart": False, "layers": 20},
        # the large grids of the benchmark: a shot from host arrays, and a run's snapshots
        {"name": "shot_cfd_4096", "kind": "advance", "method": CFD, "nx": 4096, "ny": 4096, "steps": 16, "f64": False,
         "restart": True, "layers": 0},
        {"name": "snapshot_mfd_4096", "kind": "advance", "method": MFD, "nx": 4096, "ny": 4096, "steps": 40, "f64": False,
         "restart": False, "layers": 0},
        # an ensemble of media of uneven sizes in one batch
        {"name": "batch_24", "kind": "batch", "sims": 24, "lo": 128, "hi": 1024, "steps": 16, "pick": 1},
        # requests of many sizes served from submission to their results
        {"name": "serve_6", "kind": "serve", "requests": 6, "lo": 64, "hi": 1024, "steps": 100, "pick": 1},
        # the paper's iteration on the same kind of problem
        {"name": "iterate_cfd_512", "kind": "iterate", "method": CFD, "nx": 512, "ny": 512, "steps": 2, "sweeps": 6,
         "f64": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance"] * 7 + ["batch", "serve", "static", "iterate"])
    method = rng.choice([CFD, MFD])
    if kind == "static":
        return {"kind": kind, "method": method, "nx": _log_int(rng, 16, 128), "ny": _log_int(rng, 16, 128),
                "f64": rng.random() < 0.3}
    if kind == "batch":
        return {"kind": kind, "sims": _log_int(rng, 2, 24), "lo": 64, "hi": _log_int(rng, 128, 1024),
                "steps": rng.randint(1, 16), "pick": rng.randint(2, 1000)}
    if kind == "serve":
        return {"kind": kind, "requests": rng.randint(2, 6), "lo": 64, "hi": _log_int(rng, 128, 1024),
                "steps": rng.randint(20, 100), "pick": rng.randint(2, 1000)}
    if kind == "iterate":
        return {"kind": kind, "method": method, "nx": _log_int(rng, 64, 512), "ny": _log_int(rng, 64, 512),
                "steps": rng.randint(1, 2), "sweeps": rng.randint(3, 6), "f64": rng.random() < 0.3}
    f64 = rng.random() < 0.25
    layers = 20 if rng.random() < 0.2 else 0
    hi = 1024 if f64 else 1500 if layers else 4096
    if not f64 and not layers and rng.random() < 0.15:  # a long section: lines longer than one block's chunks
        nx, ny = rng.randint(4400, 8192), _log_int(rng, 128, 1500)
        if rng.random() < 0.5:
            nx, ny = ny, nx
    else:
        nx = _log_int(rng, 32, hi)
        ny = max(32, min(hi, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    restart = method == CFD and not layers or rng.random() < 0.3
    return {"kind": kind, "method": method, "nx": nx, "ny": ny, "steps": rng.randint(1, 20 if f64 else 16 if method == CFD else 40),
            "f64": f64, "restart": restart, "layers": layers}


# ---- inputs -------------------------------------------------------------------------------------------------
H = 5.0  # cell side in metres (seismic grids)


def _shapes(method, nx, ny):
    if method == CFD:
        return ((ny + 1, nx + 1),) * 3
    return (ny + 2, nx + 2), (ny + 2, nx + 1), (ny + 1, nx + 2)


def _axis(method, n, nodes):
    """Unit coordinates of a side's points: nodes, or cell centres with the two walls."""
    if method == CFD or nodes:
        return np.arange(n + 1) / n
    return np.concatenate(([0.0], (np.arange(n) + 0.5) / n, [1.0]))


def _problem(method, nx, ny, seed):
    """A layered medium with a smooth perturbation, and fields of a few standing modes of at least 12 cells a wavelength,
    zero on the walls."""
    rng = np.random.default_rng(seed)
    x, y = _axis(method, nx, False), _axis(method, ny, False)
    speeds = np.sort(rng.uniform(1500.0, 4500.0, size=int(rng.integers(3, 7))))
    layer = np.minimum((y * speeds.size).astype(int), speeds.size - 1)
    gx = np.exp(-((x - rng.uniform(0.25, 0.75)) ** 2) / 0.02)
    gy = np.exp(-((y - rng.uniform(0.25, 0.75)) ** 2) / 0.02)
    c = speeds[layer][:, None] * (1.0 + 0.1 * np.outer(gy, gx))
    dt = (0.91 if method == CFD else 0.81) * H / float(c.max())
    U, V, W = (np.zeros(s) for s in _shapes(method, nx, ny))
    xn, yn = _axis(method, nx, True), _axis(method, ny, True)
    for _ in range(3):
        kx, ky = (math.pi * int(rng.integers(1, max(2, n // 6))) for n in (nx, ny))
        a, b = rng.uniform(0.3, 1.0), rng.uniform(-1.0, 1.0) / 3000.0
        U += a * np.outer(np.sin(ky * y), np.sin(kx * x))
        V += b * np.outer(np.sin(ky * y), np.cos(kx * xn))
        W += b * np.outer(np.cos(ky * yn), np.sin(kx * x))
    for e in (np.s_[0], np.s_[-1], np.s_[:, 0], np.s_[:, -1]):
        U[e] = 0.0
    src = (int(rng.integers(ny // 4 + 1, 3 * ny // 4)), int(rng.integers(nx // 4 + 1, 3 * nx // 4)),
           float(rng.uniform(0.5, 2.0)) * H * H / dt, 15.0, 1.2 / 15.0 * float(rng.uniform(0.0, 0.2)))
    return c, dt, U, V, W, src


def _members(case):
    """Sizes and schemes of a batch's members or a server's requests."""
    rng = np.random.default_rng(case["pick"])
    out = []
    for k in range(case.get("sims") or case["requests"]):
        if case["kind"] == "batch":
            nx, ny = (int(rng.integers(case["lo"], case["hi"] + 1)) for _ in range(2))
            steps = case["steps"]
        else:
            nx = ny = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
            # the nodal scheme's growth bounds its steps
            steps = max(1, int(rng.integers(case["steps"] // 2, case["steps"] + 1)) // (1 if k % 2 else 4))
        out.append((MFD if k % 2 else CFD, nx, ny, steps))
    return out


def _host(arrays, f64):
    """Pinned host copies, as numpy arrays."""
    return [torch.from_numpy(a).to(torch.float64 if f64 else torch.float32).pin_memory().numpy() for a in arrays]


def _empty(shapes, f64):
    return [torch.zeros(s, dtype=torch.float64 if f64 else torch.float32, pin_memory=True).numpy() for s in shapes]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        members = _members(case)
        problems = [_problem(m, nx, ny, (seed, k)) for k, (m, nx, ny, _) in enumerate(members)]
        if kind == "serve":
            return {"case": case, "members": members, "problems": problems}
        sims, shapes = [], []
        for (m, nx, ny, _), (c, dt, U, V, W, src) in zip(members, problems):
            s = adi.Sim(m, nx, ny, H, dt, c, U, V, W)
            s.set_source(*src)
            sims.append(s)
            shapes.append(s.shapes)
        # one pinned array per field for all members, and each member's view of it
        flat = _empty([sum(math.prod(sh[f]) for sh in shapes) for f in range(3)], False)
        views = [[] for _ in sims]
        for f in range(3):
            at = 0
            for k, sh in enumerate(shapes):
                n = math.prod(sh[f])
                views[k].append(flat[f][at:at + n].reshape(sh[f]))
                at += n
        return {"case": case, "sims": sims, "batch": adi.Batch(sims), "flat": flat, "views": views}
    method, nx, ny, f64 = case["method"], case["nx"], case["ny"], case["f64"]
    c, dt, U, V, W, src = _problem(method, nx, ny, seed)
    if kind == "iterate":
        return {"case": case, "dt": dt, "c": c, "fields": (U, V, W), "src": src}
    if kind == "static":
        dev = [torch.from_numpy(a).to("cuda", torch.float64 if f64 else torch.float32) for a in (c, U, V, W)]
        return {"case": case, "dt": dt, "dev": dev, "out": [torch.empty_like(a) for a in dev[1:]]}
    sim = adi.Sim(method, nx, ny, H, dt, c, U, V, W, precision=adi.ADI_FP64 if f64 else adi.ADI_FP32)
    sim.set_source(*src)
    if case["layers"]:
        sim.set_sponge(case["layers"], 0.03)
    return {"case": case, "sim": sim, "start": _host((U, V, W), f64) if case["restart"] else None,
            "out": _empty(sim.shapes, f64)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "advance":
        sim, out, f64 = state["sim"], state["out"], case["f64"]
        if state["start"] is not None:
            (sim.set_fields if f64 else sim.set_fields_f32)(*state["start"])
        sim.step(case["steps"])
        (sim.read_into if f64 else sim.read_into_f32)(*out)
        return out
    if kind == "batch":
        state["batch"].step(case["steps"])
        for sim, v in zip(state["sims"], state["views"]):
            sim.read_into_f32(*v)
        return state["flat"]
    if kind == "serve":
        srv = adi.Server(8 << 30, quantum=20)
        tickets = [srv.submit(m, nx, ny, H, dt, c, steps, U, V, W, source=src)
                   for (m, nx, ny, steps), (c, dt, U, V, W, src) in zip(state["members"], state["problems"])]
        while any(srv.tick()):
            pass
        out = [srv.result(t) for t in tickets]
        srv.close()
        return out
    if kind == "static":
        adi.step_static(case["method"], case["nx"], case["ny"], H, state["dt"],
                        adi.ADI_FP64 if case["f64"] else adi.ADI_FP32, *[t.data_ptr() for t in state["dev"] + state["out"]],
                        stream=torch.cuda.current_stream().cuda_stream)
        return state["out"]
    out = adi.fixed_point(case["method"], case["nx"], case["ny"], H, state["dt"], state["c"], *state["fields"],
                          case["steps"], source=state["src"], kmax=case["sweeps"], eps=0.0,
                          precision=adi.ADI_FP64 if case["f64"] else adi.ADI_FP32)
    return list(out[:3])


def work(case):
    """A step reads and writes the three fields once and reads the wave speed: 7 words a point; loading and reading fields
    move each value once more.  Per point and step about 60 operations solve the two line systems (block forward and
    backward substitution) or, for the iteration, about 20 a sweep."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        members = [(nx * ny, steps) for _, nx, ny, steps in _members(case)]
    else:
        members = [(case["nx"] * case["ny"], case.get("steps", 1))]
    w = 8 if case.get("f64") else 4
    moved = {"advance": 3 + 3 * bool(case.get("restart")), "batch": 3, "serve": 8, "static": 0, "iterate": 7}[kind]
    per = 40 * case["sweeps"] if kind == "iterate" else 60
    return {"bytes": float(sum(n * w * (7 * s + moved) for n, s in members)), "flops": float(sum(n * s * per for n, s in members))}


# ---- the same steps in 64 bits ------------------------------------------------------------------------------
# Peaceman-Rachford steps with the stage systems u + alpha Dv v = a, v + beta Du u = v0 solved by iterating them in
# turn (they contract), on whole arrays; the compact operators' tridiagonal systems by cyclic reduction.
D_END = [-4751 / 5192, 909 / 1298, 6091 / 15576, -1165 / 5192, 129 / 2596, -25 / 15576]
G_END = [-47888 / 14245, 1790 / 407, -14545 / 9768, 8997 / 16280, -2335 / 22792, 25 / 9768]
G_NEXT = [16 / 105, -31 / 24, 29 / 24, -3 / 40, 1 / 168]
W4 = [1 / 24, -9 / 8, 9 / 8, -1 / 24]


def _dot(x, weights, first):
    return sum(w * x[..., first + k] for k, w in enumerate(weights))


def _tri(lo, di, up, dev):
    """Reduction steps (shift, a, c) and the last diagonal of a tridiagonal matrix: r_i <- r_i + a_i r_{i-s} + c_i r_{i+s}."""
    lo, di, up = (np.array(v, dtype=np.float64) for v in (lo, di, up))
    n, s, steps = len(di), 1, []
    while s < n and max(np.abs(lo).max(), np.abs(up).max()) > 1e-22:
        a, c, l2, u2, d2 = np.zeros(n), np.zeros(n), np.zeros(n), np.zeros(n), di.copy()
        a[s:] = -lo[s:] / di[:-s]
        c[:-s] = -up[:-s] / di[s:]
        l2[s:] = a[s:] * lo[:-s]
        u2[:-s] = c[:-s] * up[s:]
        d2[s:] += a[s:] * up[:-s]
        d2[:-s] += c[:-s] * lo[s:]
        steps.append((s, torch.tensor(a, device=dev), torch.tensor(c, device=dev)))
        lo, di, up, s = l2, d2, u2, 2 * s
    return steps, torch.tensor(1.0 / di, device=dev)


def _tri_solve(f, r):
    for s, a, c in f[0]:
        q = r.clone()
        q[..., s:].addcmul_(a[s:], r[..., :-s])
        q[..., :-s].addcmul_(c[:-s], r[..., s:])
        r = q
    return r * f[1]


class _Line:
    """Du and Dv along the last axis, N cells of side H."""

    def __init__(self, method, N, dev):
        self.method, self.N = method, N
        if method == CFD:
            lo, di, up = np.ones(N + 1), np.full(N + 1, 4.0), np.ones(N + 1)
            lo[0] = up[N] = 0.0
            di[0] = di[N] = 6.0
            up[0] = lo[N] = 18.0
            self.P = _tri(lo, di, up, dev)
            lo, di, up = np.ones(N - 1), np.full(N - 1, 4.0), np.ones(N - 1)
            lo[0] = up[-1] = 0.0
            di[0] = di[-1] = 6.0
            up[0] = lo[-1] = 6.0
            self.B = _tri(lo, di, up, dev)

    def du(self, p):
        N = self.N
        if self.method == CFD:
            q = torch.empty_like(p)
            q[..., 1:N] = 3 * (p[..., 2:] - p[..., :-2])
            q[..., 0] = _dot(p, [-17, 9, 9, -1], 0)
            q[..., N] = _dot(p, [1, -9, -9, 17], N - 3)
            return _tri_solve(self.P, q) / H
        q = p.new_empty(p.shape[:-1] + (N + 1,))
        q[..., 2:N - 1] = sum(w * p[..., 1 + k:N - 2 + k] for k, w in enumerate(W4))
        q[..., 0], q[..., 1] = _dot(p, G_END, 0), _dot(p, G_NEXT, 0)
        q[..., N], q[..., N - 1] = -_dot(p, G_END[::-1], N - 4), -_dot(p, G_NEXT[::-1], N - 3)
        return q / H

    def dv(self, v):
        N = self.N
        if self.method == CFD:
            q = 3 * (v[..., 2:] - v[..., :-2])
            q[..., 0] = _dot(v, [-1, -9, 9, 1], 0)
            q[..., -1] = _dot(v, [-1, -9, 9, 1], N - 3)
            return _tri_solve(self.B, q) / H
        q = v.new_empty(v.shape[:-1] + (N,))
        q[..., 1:N - 1] = sum(w * v[..., k:N - 2 + k] for k, w in enumerate(W4))
        q[..., 0], q[..., -1] = _dot(v, D_END, 0), -_dot(v, D_END[::-1], N - 5)
        return q / H


def _stage(line, a, v0, u, v, alpha, beta, sweeps, tol):
    """u + alpha Dv v = a on the inner points, v + beta Du u = v0; u's ends are given.  `sweeps` plain sweeps from (u, v);
    with 0 the solution: damped sweeps (the plain ones' factors lie between -1 and 0, the damped ones' within 1/3)."""
    u = u.clone()
    if not sweeps:
        v = v0 - beta * line.du(u)
    for k in range(sweeps or 100):
        change = a - alpha * line.dv(v) - u[..., 1:-1]
        u[..., 1:-1] += change if sweeps else change * (2 / 3)
        v = v0 - beta * line.du(u)
        if not sweeps and k % 8 == 7 and bool(change.abs().max() <= tol * u.abs().max()):
            break
    return u, v


def _steps64(method, nx, ny, dt, c, U, V, W, steps, src, layers=0, sweeps=0, tol=1e-15):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    c, U, V, W = (torch.tensor(a, dtype=torch.float64, device=dev) for a in (c, U, V, W))
    X, Y = _Line(method, nx, dev), _Line(method, ny, dev)
    al, beta = 0.5 * dt * c[1:-1, 1:-1] ** 2, 0.5 * dt
    T = lambda t: t.T.contiguous()  # noqa: E731
    alT = T(al)

    def forcing(t):
        if src is None:
            return 0.0
        q = (math.pi * src[3] * (t - src[4])) ** 2
        return 0.5 * dt * src[2] * (1 - 2 * q) * math.exp(-q) / (H * H)

    damp = None
    if layers:
        def side(n, nodes):
            x = torch.tensor(_axis(method, n, nodes) * n, device=dev)
            return torch.minimum(x, n - x)
        damp = []
        for ys, xs in ((False, False), (False, True), (True, False)):
            d = torch.minimum(side(ny, ys)[:, None], side(nx, xs)[None, :])
            damp.append(torch.exp(-(0.03 * (layers - d).clamp(min=0.0)) ** 2))
        for e in (np.s_[0], np.s_[-1], np.s_[:, 0], np.s_[:, -1]):
            damp[0][e] = 1.0
    for m in range(steps):
        ui, wi = T(U[:, 1:-1]), T(W[:, 1:-1])  # y-lines
        a = U[1:-1, 1:-1] - al * T(Y.dv(wi))
        if src is not None:
            a[src[0] - 1, src[1] - 1] += forcing(m * dt)
        ws = wi - beta * Y.du(ui)
        us, vs = _stage(X, a, V[1:-1], U[1:-1], V[1:-1], al, beta, sweeps, tol)
        C = T(us[:, 1:-1] - al * X.dv(vs))
        if src is not None:
            C[src[1] - 1, src[0] - 1] += forcing((m + 1) * dt)
        V = V.clone()
        V[1:-1] = vs - beta * X.du(us)
        u0 = ui.clone()
        u0[:, 1:-1] = T(us[:, 1:-1])
        u2, w2 = _stage(Y, C, ws, u0, wi, alT, beta, sweeps, tol)
        U, W = U.clone(), W.clone()
        U[:, 1:-1], W[:, 1:-1] = T(u2), T(w2)
        if damp is not None:
            U, V, W = U * damp[0], V * damp[1], W * damp[2]
    return [U, V, W]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        members = _members(case)
        res = [_steps64(m, nx, ny, p[1], p[0], *_as_held(p, True), steps, p[5], tol=1e-13)
               for k, (m, nx, ny, steps) in enumerate(members) for p in [_problem(m, nx, ny, (seed, k))]]
        return res if kind == "serve" else [torch.cat([r[f].reshape(-1) for r in res]) for f in range(3)]
    method, nx, ny, f64 = case["method"], case["nx"], case["ny"], case["f64"]
    p = _problem(method, nx, ny, seed)
    c, dt, fields, src = p[0], p[1], _as_held(p, f64 or not case.get("restart")), p[5]
    if kind == "iterate":
        return _steps64(method, nx, ny, dt, c, *fields, case["steps"], src, sweeps=case["sweeps"])
    if kind == "static":
        held = lambda a: a if f64 else a.astype(np.float32).astype(np.float64)  # noqa: E731
        return _steps64(method, nx, ny, dt, held(c), *[held(a) for a in fields], 1, None)
    return _steps64(method, nx, ny, dt, c, *fields, case["steps"], src, layers=case["layers"], tol=1e-15 if f64 else 1e-13)


def _as_held(p, whole):
    """The start's fields as the caller passes them: in 64 bits, or rounded to 32 bits first."""
    return [a if whole else a.astype(np.float32).astype(np.float64) for a in p[2:5]]
