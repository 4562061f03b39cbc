"""The solver's workloads as timed cases: whole steps (a new geometry, then its solve), batches,
a request stream, single multigrid cycles and the coefficient build, each through the library's
public entry points.

Sizes are those of the benchmark's and the tests' configurations (129^2 sine warp, 1025^2
inclusion, 8193^2 annulus, uneven batches of 65-513, requests of 129-1025) and generic ones of
the form m 2^k + 1.  Every input is a function of the seed alone.  ``exact`` computes the same
outputs in FP64 with torch, from the discretization's formulas.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2602_01888_gb300 import inputs as I
from paper_2602_01888_gb300 import mg

DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest problem a user solves: resident 129^2 sine-warp grid, plain FP64 V(2,2) cycles
        {"name": "solve_warp_129_fp64", "kind": "solve", "map": "warp", "nx": 129, "ny": 129,
         "prec": "fp64", "outer": "vcycle", "smoother": "gs4", "nu": 2, "rtol": 1e-10, "update": False},
        # one small request: new inclusion geometry and material, mixed-precision solve
        {"name": "step_inclusion_257_mixed", "kind": "solve", "map": "inclusion", "nx": 257, "ny": 257,
         "prec": "mixed", "outer": "fcg", "smoother": "gs4", "nu": 2, "rtol": 1e-9, "update": True},
        # the 1025^2 inclusion benchmark, both precisions
        {"name": "step_inclusion_1025_fp64", "kind": "solve", "map": "inclusion", "nx": 1025, "ny": 1025,
         "prec": "fp64", "outer": "fcg", "smoother": "gs4", "nu": 2, "rtol": 3e-8, "update": True},
        {"name": "step_inclusion_1025_mixed", "kind": "solve", "map": "inclusion", "nx": 1025, "ny": 1025,
         "prec": "mixed", "outer": "fcg", "smoother": "gs4", "nu": 2, "rtol": 3e-8, "update": True},
        # the annulus benchmark: line smoother, FP64 at a medium size and the 8193^2 headline
        {"name": "step_annulus_4097_fp64_line", "kind": "solve", "map": "polar", "nx": 4097, "ny": 4097,
         "prec": "fp64", "outer": "fcg", "smoother": "xline", "nu": 1, "rtol": 2e-9, "update": True},
        {"name": "step_annulus_8193_mixed_line", "kind": "solve", "map": "polar", "nx": 8193, "ny": 8193,
         "prec": "mixed", "outer": "fcg", "smoother": "xline", "nu": 1, "rtol": 1e-8, "update": True},
        # the batched workload: uneven instances (sides 65-513), rebuilt and solved together
        {"name": "batch_64_mixed", "kind": "batch", "count": 64, "mix": 4000, "lo": 65, "hi": 513, "prec": "mixed", "rtol": 1e-9},
        # the serving loop: host arrays submitted together, results polled
        {"name": "serve_24_mixed", "kind": "serve", "count": 24, "mix": 5, "lo": 129, "hi": 1025, "rtol": 1e-9},
        # single cycles on a caller's hierarchy, as an outer solver would call them
        {"name": "cycle_point_f32_4097x2049", "kind": "cycle", "nx": 4097, "ny": 2049, "prec": "f32", "line": False, "nu": 2},
        {"name": "cycle_point_f64_1537x1025", "kind": "cycle", "nx": 1537, "ny": 1025, "prec": "f64", "line": False, "nu": 2},
        {"name": "cycle_line_f32_3073x1537", "kind": "cycle", "nx": 3073, "ny": 1537, "prec": "f32", "line": True, "nu": 1},
        # the coefficient build by single entry points: mapped grid -> tensor -> operator -> two coarse levels
        {"name": "build_grid_2049_f64", "kind": "build", "nx": 2049, "ny": 2049},
    ]


def _snap(v):
    """Nearest m 2^k + 1 with 8 <= m <= 16 and, so that the two sides may differ by a factor of a few
    and still share a hierarchy, k >= 3."""
    return min((m * 2 ** k + 1 for k in range(3, 10) for m in range(8, 17)), key=lambda s: abs(s - v))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _pair(rng, lo, hi):
    """Two sides m 2^k + 1 of the same k (so the coarsest level stays small), within [lo, hi]."""
    n = _snap(_log(rng, lo, hi))
    k = ((n - 1) & -(n - 1)).bit_length() - 1
    while (n - 1) >> k < 8:
        k -= 1
    return n, rng.randint(8, 16) * 2 ** k + 1


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        c = _draw(rng)
        if c not in known:
            return c


def _draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "annulus", "batch", "serve", "cycle", "cycle", "build"])
    if kind == "solve":
        m = rng.choice(["warp", "affine", "sinh", "inclusion", "inclusion", "semi"])
        n = _snap(_log(rng, 129, 2049))
        nx, ny = (n, n) if m in ("inclusion", "sinh", "semi") else _pair(rng, 129, 2049)
        # the semi-annulus needs the line smoother; the others take the default
        return {"kind": "solve", "map": m, "nx": nx, "ny": ny, "prec": rng.choice(["fp64", "mixed", "mixed"]),
                "outer": rng.choice(["fcg", "fcg", "vcycle"]) if m not in ("inclusion", "sinh") else "fcg",
                "smoother": "xline" if m == "semi" else "gs4", "nu": 1 if m == "semi" else 2,
                "rtol": 1e-9, "update": rng.random() < 0.7}
    if kind == "annulus":
        n = _snap(_log(rng, 257, 8000))
        # FP64 stops above the residual floor of the larger grids, and stays under the largest listed cost
        prec = rng.choice(["fp64", "mixed"]) if n <= 4097 else "mixed"
        return {"kind": "solve", "map": "polar", "nx": n, "ny": n, "prec": prec, "outer": "fcg",
                "smoother": "xline", "nu": rng.randint(1, 2) if n <= 2049 else 1,
                "rtol": 2e-9 if n <= 4097 else 1e-8, "update": True}
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 4, 64), "mix": rng.randrange(1000), "lo": 65, "hi": rng.choice([129, 257, 513]),
                "prec": rng.choice(["fp64", "mixed", "mixed"]), "rtol": 1e-9}
    if kind == "serve":
        return {"kind": "serve", "count": _log(rng, 6, 24), "mix": rng.randrange(1000), "lo": 129, "hi": rng.choice([257, 513, 1025]), "rtol": 1e-9}
    if kind == "cycle":
        prec = rng.choice(["f32", "f64"])
        nx, ny = _pair(rng, 193, 2049 if prec == "f64" else 4097)
        ny = min(ny, 4097 if prec == "f32" else 2049)
        k = min(((nx - 1) & -(nx - 1)), ((ny - 1) & -(ny - 1)))
        if max(nx - 1, ny - 1) // k > 16:
            ny = nx
        return {"kind": "cycle", "nx": nx, "ny": ny, "prec": prec, "line": rng.random() < 0.5, "nu": rng.randint(1, 2)}
    nx, ny = _pair(rng, 129, 2049)
    return {"kind": "build", "nx": nx, "ny": min(ny, 2049) if min(ny, 2049) % 4 == 1 else nx}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return np.random.default_rng(seed)


def _coords(g):
    x = g.x0 + g.hx * torch.arange(g.nx, dtype=F64, device=DEV)
    y = g.y0 + g.hy * torch.arange(g.nyr, dtype=F64, device=DEV)
    return x[None, :].expand(g.nyr, g.nx), y[:, None].expand(g.nyr, g.nx)


def _inclusion_map(n, i0):
    """Mapped coordinates of the unit square with a disc of the inner square's half-width: the square's
    concentric shells go to circles inside (Eq. 44 scaled by the shell) and blend linearly from the
    disc's edge to the outer square outside."""
    g = I.Grid(n, n)
    x, y = _coords(g)
    u, v = x - 0.5, y - 0.5
    r = 0.5 - i0 / (n - 1)
    rho = torch.maximum(u.abs(), v.abs())
    safe = torch.where(rho > 0, rho, torch.ones_like(rho))
    su, sv = u / safe, v / safe  # the direction, a point of the unit square's boundary
    on_y = sv.abs() >= su.abs()
    bx = torch.where(on_y, su / math.sqrt(2.0), torch.sign(su) * torch.sqrt((1 - sv * sv / 2).clamp(min=0)))
    by = torch.where(on_y, torch.sign(sv) * torch.sqrt((1 - su * su / 2).clamp(min=0)), sv / math.sqrt(2.0))
    t = ((rho - r) / (0.5 - r)).clamp(min=0)
    inside = torch.minimum(rho, torch.full_like(rho, r))
    xp = 0.5 + torch.where(rho > r, (1 - t) * r * bx + t * 0.5 * su, inside * bx)
    yp = 0.5 + torch.where(rho > r, (1 - t) * r * by + t * 0.5 * sv, inside * by)
    return xp.contiguous(), yp.contiguous()


def _blobs(xp, yp, rng, count=16, sigma=0.02):
    cx, cy, amp = rng.uniform(0, 1, count), rng.uniform(0, 1, count), rng.uniform(-1, 1, count)
    rho = torch.zeros_like(xp)
    for k in range(count):
        rho += float(amp[k]) * torch.exp(-((xp - float(cx[k])) ** 2 + (yp - float(cy[k])) ** 2) / (2 * sigma * sigma))
    return rho


def _waves(xp, yp, rng, modes):
    rho = torch.zeros_like(xp)
    for _ in range(modes):
        kx, ky = (int(v) for v in rng.integers(-8, 9, 2))
        kk = max(1.0, math.hypot(kx, ky))
        rho += float(rng.standard_normal()) / kk ** 2 * torch.cos(
            math.pi * (kx * xp + ky * yp) + float(rng.uniform(0, 2 * math.pi)))
    return rho


def _inclusion(n, rng):
    """(xp, yp, eps', rho') of one inclusion instance: radius U[0.1, 0.35] on a grid line, ratio U[2, 50]."""
    i0 = I.snap_ring(n, float(rng.uniform(0.1, 0.35)))
    xp, yp = _inclusion_map(n, i0)
    ratio = float(rng.uniform(2.0, 50.0))
    eps = torch.ones(n, n, dtype=F64, device=DEV)
    i1 = n - 1 - i0
    eps[i0:i1 + 1, i0:i1 + 1] = 0.5 * (1 + ratio)
    eps[i0 + 1:i1, i0 + 1:i1] = ratio
    return xp, yp, eps, _blobs(xp, yp, rng)


def _instance(case, seed):
    """Grid, map and device arrays of a 'solve' case: dict with g, spec, xp, yp, eps, rho, bc."""
    rng = _gen(seed)
    nx, ny, m = case["nx"], case["ny"], case["map"]
    d = {"xp": None, "yp": None, "eps": None, "bc": None}
    if m == "inclusion":
        g, spec = I.Grid(nx, ny), I.MapSpec("grid")
        d["xp"], d["yp"], d["eps"], rho = _inclusion(nx, rng)
    else:
        if m == "polar":
            g, spec = I.annulus_grid(nx), I.MapSpec("polar")
        elif m == "semi":  # half annulus, insulated straight sides, potential given on the arcs
            g, spec = I.Grid(nx, ny, 2.0, 0.0, 3.0, math.pi, neumann_y=True), I.MapSpec("polar")
        elif m == "sinh":
            g, spec = I.Grid(nx, ny, -3.0, -3.0, 6.0, 6.0), I.MapSpec("sinh", (5.0, float(rng.uniform(0.5, 0.6))))
        elif m == "warp":
            g = I.Grid(nx, ny, 0.0, 0.0, 1.0, (ny - 1) / (nx - 1) if ny != nx else 1.0)
            spec = I.MapSpec("sine_warp", (float(rng.uniform(0.03, 0.1)),))
        else:
            g = I.Grid(nx, ny, 0.0, 0.0, 1.0, (ny - 1) / (nx - 1))
            spec = I.MapSpec("affine", (1.0, float(rng.uniform(0.1, 0.4)), -0.2, 1.1))
        x, y = _coords(g)
        if spec.kind == "polar":
            px, py = x * torch.cos(y), x * torch.sin(y)
        elif spec.kind == "sinh":
            px, py = 5.0 * torch.sinh(spec.params[1] * x), 5.0 * torch.sinh(spec.params[1] * y)
        else:
            px, py = x, y
        if m == "sinh":  # a beam at the origin, held at a smooth potential on the boundary
            s = float(rng.uniform(0.4, 1.0))
            rho = -100.0 * torch.exp(-(px * px + py * py) / (2 * s * s))
            d["bc"] = torch.log(1.0 + px * px + py * py).contiguous()
        elif m == "semi":
            rho = _waves(px, py, rng, 8)
            d["bc"] = torch.where(x < 3.5, float(rng.uniform(0.5, 2.0)), 0.0).to(F64).contiguous()
        elif m == "affine":
            rho = _waves(px, py, rng, 8)
            d["bc"] = (px * px + float(rng.uniform(0.5, 1.5)) * py).contiguous()
        else:
            rho = _waves(px, py, rng, 16)
    return dict(d, g=g, spec=spec, rho=rho.contiguous())


def _sides(case):
    """The case's sides: the batch's powers of two plus one, the requests' log-uniform m 2^k + 1."""
    rng, count, lo, hi = _gen(case["mix"]), case["count"], case["lo"], case["hi"]
    if case["kind"] == "batch":
        return [int(v) for v in rng.choice([s for s in (65, 129, 257, 513) if lo <= s <= hi], count)]
    return [min(hi, I.snap_side(math.exp(rng.uniform(math.log(lo), math.log(hi))))) for _ in range(count)]


_contexts = []


def _ctx():
    """One library context for the process, as a program keeps it."""
    if not _contexts:
        _contexts.append(mg.Context(0))
    return _contexts[0]


class _Problem:
    """A resident problem built from device arrays, freed with the state."""

    def __init__(self, g, spec, eps, opts, xp, yp):
        self.ctx = _ctx()
        self.h = mg.mg_setup_transform(self.ctx.h, g, spec, eps, opts, xp, yp)

    def __del__(self):
        if getattr(self, "h", None) and self.ctx.h:  # a closed context has already freed it
            mg.mg_problem_free(self.h)


class _Server:
    """A request server on a context of its own, stopped when the state goes."""

    def __init__(self):
        self.ctx = mg.Context(0)
        self.h = mg.mg_server_start(self.ctx.h, max_inflight=16)

    def __del__(self):
        try:
            mg.mg_server_stop(self.h)
            self.ctx.close()
        except Exception:
            pass


def _opts(case):
    return mg.make_opts(case.get("prec", "mixed"), case.get("outer", "fcg"), rtol=case["rtol"], max_iters=400,
                        nu1=case.get("nu", 2), nu2=case.get("nu", 2), smoother=case.get("smoother", "gs4"))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        s = _instance(case, seed)
        s["opts"], s["update"] = _opts(case), case["update"]
        torch.cuda.synchronize()
        s["prob"] = _Problem(s["g"], s["spec"], s["eps"], s["opts"], s["xp"], s["yp"])
        s["phi"] = torch.zeros(s["g"].shape, dtype=F64, device=DEV)
    elif kind == "batch":
        rng = _gen(seed)
        s = {"opts": _opts(case), "g": [], "xp": [], "yp": [], "eps": [], "rho": [], "phi": [], "prob": []}
        for n in _sides(case):
            xp, yp, eps, rho = _inclusion(n, rng)
            for k, v in (("g", I.Grid(n, n)), ("xp", xp), ("yp", yp), ("eps", eps), ("rho", rho), ("phi", torch.zeros_like(rho))):
                s[k].append(v)
        torch.cuda.synchronize()
        s["spec"] = [I.MapSpec("grid")] * case["count"]
        for g, xp, yp, eps in zip(s["g"], s["xp"], s["yp"], s["eps"]):
            s["prob"].append(_Problem(g, s["spec"][0], eps, s["opts"], xp, yp))
    elif kind == "serve":
        rng = _gen(seed)
        s = {"opts": _opts(case), "req": []}
        for n in _sides(case):
            xp, yp, eps, rho = (v.cpu().numpy() for v in _inclusion(n, rng))
            s["req"].append((I.Grid(n, n), I.MapSpec("grid", (), xp, yp), rho, eps, np.zeros((n, n))))
        s["server"] = _Server()
    elif kind == "cycle":
        s = _hierarchy(case, seed)
    else:
        s = _build_state(case, seed)
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    if "server" in s:
        t = []
        for g, spec, rho, eps, _ in s["req"]:
            rc, ticket = mg.mg_serve_submit(s["server"].h, g, spec, rho, None, eps, s["opts"])
            if rc != mg.MG_OK:
                raise RuntimeError(f"submit: status {rc}")
            t.append(ticket)
        for ticket, (_, _, _, _, phi) in zip(t, s["req"]):
            rc, _ = mg.mg_serve_poll(s["server"].h, ticket, 60000, phi)
            if rc != mg.MG_OK:
                raise RuntimeError(f"poll: status {rc}")
        return [r[4] for r in s["req"]]
    if "levels" in s:
        return _cycle_run(s)
    if "fine" in s:
        return _build_run(s)
    if isinstance(s["prob"], list):
        h = [p.h for p in s["prob"]]
        mg.mg_batch_update_transform(_ctx().h, h, s["spec"], s["eps"], s["xp"], s["yp"])
        mg.mg_batch_solve(_ctx().h, h, s["rho"], None, s["phi"], s["opts"])
        return s["phi"]
    if s["update"]:
        mg.mg_update_transform(s["prob"].h, s["g"], s["spec"], s["eps"], s["xp"], s["yp"])
    mg.mg_solve(s["prob"].h, s["rho"], s["bc"], s["phi"], s["opts"])
    return s["phi"]


# ------------------------------------------------------------------ single cycles
def _pitch(nx):
    return (nx + 31) // 32 * 32


def _pitched(a, dt):
    out = torch.zeros(a.shape[0], _pitch(a.shape[1]), dtype=dt, device=DEV)
    out[:, :a.shape[1]] = a
    return out


def _cycle_operators(case, seed):
    """FP64 operators of a sine-warp hierarchy whose coarse levels are the map's own discretization on
    each coarse grid, and the right-hand side (interior nodes, residual-sized)."""
    rng = _gen(seed)
    nx, ny = case["nx"], case["ny"]
    spec = I.MapSpec("sine_warp", (float(rng.uniform(0.03, 0.09)),))
    ops = []
    while True:
        g = I.Grid(nx, ny, 0.0, 0.0, 1.0, (case["ny"] - 1) / (case["nx"] - 1))
        ops.append(_Op(g, *_tensor(g, spec)[1:]))
        if (nx - 2) * (ny - 2) <= 64 or (nx - 1) % 2 or (ny - 1) % 2 or min(nx, ny) < 5:
            break
        nx, ny = (nx - 1) // 2 + 1, (ny - 1) // 2 + 1
    t = torch.Generator(device=DEV)
    t.manual_seed(int(seed))
    b = torch.randn(ops[0].E.shape, dtype=F64, device=DEV, generator=t) * ops[0].mask * ops[0].diag.max()
    return ops, b


def _hierarchy(case, seed):
    f32 = case["prec"] == "f32"
    dt = torch.float32 if f32 else F64
    ops, b = _cycle_operators(case, seed)
    s = {"levels": len(ops), "f32": f32, "line": case["line"], "nu": case["nu"], "nx": case["nx"], "keep": [],
         "x": [], "b": [], "t": [], "f": []}
    s["ops"] = ((mg.mgk_op_f32 if f32 else mg.mgk_op_f64) * len(ops))()
    tag, st = case["prec"], mg._stream()
    for l, A in enumerate(ops):
        arr = [_pitched(v, dt) for v in (A.E, A.N, A.NE, A.NW, A.diag)]
        arr.append((1.0 / arr[4].clamp(min=1e-30)).contiguous())
        s["keep"].append(arr)
        s["ops"][l] = mg.op_struct(arr, A.nx, A.ny, False, f32=f32)
        s["x"].append(torch.zeros_like(arr[0]))
        s["b"].append(_pitched(b, dt) if l == 0 else torch.zeros_like(arr[0]))
        s["t"].append(torch.zeros_like(arr[0]))
        if case["line"] and l < len(ops) - 1:
            f = torch.zeros(mg.lib().mgk_line_factor_elems(A.nx, A.ny, 0), dtype=dt, device=DEV)
            mg.mgk("mgk_line_factor_" + tag, C.byref(s["ops"][l]), f.data_ptr(), st)
            s["f"].append(f)
    A = ops[-1]
    m = (A.nx - 2) * (A.ny - 2)
    s["inv"] = torch.zeros(m * m, dtype=F64, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    arr = [v.double() for v in s["keep"][-1]]
    mg.mgk("mgk_coarse_factor", C.byref(mg.op_struct(arr, A.nx, A.ny, False)), s["inv"].data_ptr(), status.data_ptr(), st)
    for k in ("x", "b", "t", "f"):
        s["p" + k] = (C.c_void_p * max(1, len(s[k])))(*[v.data_ptr() for v in s[k]])
    torch.cuda.synchronize()
    return s


def _cycle_run(s):
    s["x"][0].zero_()  # the cycle as a preconditioner: it starts from zero
    tag = "f32" if s["f32"] else "f64"
    if s["line"]:
        mg.mgk("mgk_vcycle_line_" + tag, s["levels"], s["ops"], s["px"], s["pb"], s["pt"], s["inv"].data_ptr(), s["pf"],
               s["nu"], s["nu"], mg._stream())
    else:
        mg.mgk("mgk_vcycle_" + tag, s["levels"], s["ops"], s["px"], s["pb"], s["pt"], s["inv"].data_ptr(), s["nu"],
               s["nu"], 0, mg._stream())
    return s["x"][0][:, :s["nx"]]


# ------------------------------------------------------------------ coefficient build
def _build_state(case, seed):
    """A smooth mapped grid with a varying material, and the arrays a caller keeps for its operators."""
    rng = _gen(seed)
    g = I.Grid(case["nx"], case["ny"])
    x, y = _coords(g)
    a, b = (float(v) for v in rng.uniform(0.03, 0.08, 2))
    xp = _pitched(x + a * torch.sin(math.pi * x) * torch.sin(2 * math.pi * y), F64)
    yp = _pitched(y + b * torch.sin(2 * math.pi * x) * torch.sin(math.pi * y), F64)
    eps = _pitched(torch.exp(_waves(x, y, rng, 4)), F64)
    s = {"g": g, "xp": xp, "yp": yp, "eps": eps, "tensor": [torch.zeros_like(xp) for _ in range(4)],
         "folded": torch.zeros(1, dtype=torch.int32, device=DEV), "fine": [], "ops": []}
    nx, ny = g.nx, g.ny
    for _ in range(3):
        arr = [torch.zeros(ny, _pitch(nx), dtype=F64, device=DEV) for _ in range(6)]
        s["fine"].append(arr)
        s["ops"].append(mg.op_struct(arr, nx, ny, False))
        nx, ny = (nx - 1) // 2 + 1, (ny - 1) // 2 + 1
    return s


def _build_run(s):
    g, st, t = s["g"], mg._stream(), s["tensor"]
    mg.mgk("mgk_eps_grid", g.nx, g.ny, 0, g.hx, g.hy, s["xp"].data_ptr(), s["yp"].data_ptr(), 0.0, 0.0, s["eps"].data_ptr(),
           s["xp"].shape[1], *[v.data_ptr() for v in t], s["folded"].data_ptr(), st)
    mg.mgk("mgk_assemble", C.byref(s["ops"][0]), g.hx, g.hy, *[v.data_ptr() for v in t[1:]], st)
    for l in (0, 1):
        mg.mgk("mgk_galerkin", C.byref(s["ops"][l]), C.byref(s["ops"][l + 1]), st)
    return [v[:, :g.nx] for v in t] + [v[:, :o.nx] for o, arr in zip(s["ops"], s["fine"]) for v in arr]


# ------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        # five arrays in and out a node: mapped coordinates, material, source, potential
        nodes = float(sum(n * n for n in _sides(case)))
        return {"bytes": 40.0 * nodes, "flops": 8 * 170.0 * nodes}
    nodes = float(case["nx"]) * case["ny"]
    if kind == "solve":
        arrays = 2 + (3 if case["map"] == "inclusion" else 0) + (1 if case["map"] in ("sinh", "semi", "affine") else 0)
        # about eight cycles of (nu1 + nu2 + 1) operator passes, a third more for the coarse levels
        return {"bytes": 8.0 * arrays * nodes, "flops": 8 * (2 * case["nu"] + 2) * 18 * 4 / 3 * nodes}
    if kind == "cycle":
        e = 4 if case["prec"] == "f32" else 8
        return {"bytes": 7.0 * e * nodes * 4 / 3, "flops": (2 * case["nu"] + 1) * 18 * 4 / 3 * nodes}
    return {"bytes": 8.0 * nodes * (3 + 4 + 6 * (1 + 1 / 4 + 1 / 16)), "flops": 60.0 * nodes + 220.0 * nodes * (1 / 4 + 1 / 16)}


# ------------------------------------------------------------------ the same in FP64 torch
def _tensor(g, spec, xp=None, yp=None, eps=None):
    """(D, eps_xx, eps_xy, eps_yy) of a map (Eqs. 10, 12-15): analytic Jacobian, or the differences of
    Eqs. 39-42 with one-sided second-order ends."""
    x, y = _coords(g)
    p = spec.params
    one, zero = torch.ones(g.shape, dtype=F64, device=DEV), torch.zeros(g.shape, dtype=F64, device=DEV)
    if spec.kind == "grid":
        def dx(f):
            d = torch.empty_like(f)
            d[:, 1:-1] = f[:, 2:] - f[:, :-2]
            d[:, 0] = -3 * f[:, 0] + 4 * f[:, 1] - f[:, 2]
            d[:, -1] = 3 * f[:, -1] - 4 * f[:, -2] + f[:, -3]
            return d
        a, c = dx(xp) * (0.5 / g.hx), dx(yp) * (0.5 / g.hx)
        b, d = dx(xp.t()).t() * (0.5 / g.hy), dx(yp.t()).t() * (0.5 / g.hy)
    elif spec.kind == "polar":
        a, b, c, d = torch.cos(y), -x * torch.sin(y), torch.sin(y), x * torch.cos(y)
    elif spec.kind == "sinh":
        a, b, c, d = p[0] * p[1] * torch.cosh(p[1] * x), zero, zero, p[0] * p[1] * torch.cosh(p[1] * y)
    elif spec.kind == "sine_warp":
        k, pi = p[0], math.pi
        a = 1 + k * pi * torch.cos(pi * x) * torch.sin(pi * y)
        b = k * pi * torch.sin(pi * x) * torch.cos(pi * y)
        c = 2 * k * pi * torch.cos(2 * pi * x) * torch.sin(pi * y)
        d = 1 + k * pi * torch.sin(2 * pi * x) * torch.cos(pi * y)
    else:
        a, b, c, d = p[0] * one, p[1] * one, p[2] * one, p[3] * one
    det = a * d - b * c
    s = (1.0 if eps is None else eps) / det
    exy = zero if spec.kind in ("polar", "sinh") else s * (-d * c - b * a)
    return det, s * (d * d + b * b), exy, s * (c * c + a * a)


class _Op:
    """The symmetric 9-point operator on a grid from its nodal tensor, or from stored couplings."""

    def __init__(self, g, exx=None, exy=None, eyy=None):
        self.nx, self.ny, self.periodic = g.nx, g.ny, g.periodic_y
        self.mask = torch.zeros(g.shape, dtype=torch.bool, device=DEV)
        (self.mask[:, 1:-1] if g.periodic_y else self.mask[1:-1, 1:-1]).fill_(True)
        if exx is None:
            return
        z = torch.zeros_like(exx)
        self.E, self.N, self.NE, self.NW = z.clone(), z.clone(), z.clone(), z.clone()
        top = slice(None) if g.periodic_y else slice(0, -1)
        self.E[:, :-1] = -0.5 * (exx[:, :-1] + exx[:, 1:]) / g.hx ** 2
        self.N[top] = (-0.5 * (eyy + self.up(eyy)) / g.hy ** 2)[top]
        q = 4 * g.hx * g.hy
        self.NE[top, :-1] = (-(exy[:, 1:] + self.up(exy)[:, :-1]) / q)[top]
        self.NW[top, 1:] = ((exy[:, :-1] + self.up(exy)[:, 1:]) / q)[top]
        s = self.E + self.w(self.E) + self.N + self.dn(self.N) + self.NE + self.dn(self.w(self.NE)) + self.NW + self.dn(self.e(self.NW))
        self.diag = torch.where(self.mask, -s, torch.ones_like(s))

    # value at the node above, below, to the right, to the left (wrapped: never used across a side)
    up = staticmethod(lambda a: torch.roll(a, -1, 0))
    dn = staticmethod(lambda a: torch.roll(a, 1, 0))
    e = staticmethod(lambda a: torch.roll(a, -1, 1))
    w = staticmethod(lambda a: torch.roll(a, 1, 1))

    def cross(self, x):
        """Couplings to the rows above and below, times x."""
        u, d = self.up(x), self.dn
        return (self.N * u + d(self.N * x) + self.NE * self.e(u) + d(self.w(self.NE * x)) + self.NW * self.w(u)
                + d(self.e(self.NW * x)))

    def off(self, x):
        return self.cross(x) + self.E * self.e(x) + self.w(self.E * x)

    def residual(self, x, b):
        return torch.where(self.mask, b - self.off(x) - self.diag * x, torch.zeros_like(b))

    def colour(self, x, b, reverse):
        """One four-colour Gauss-Seidel sweep."""
        cols = [(0, 0), (1, 1), (1, 0), (0, 1)]
        for ci, cj in cols[::-1] if reverse else cols:
            m = torch.zeros_like(self.mask)
            m[cj::2, ci::2] = True
            x = torch.where(m & self.mask, (b - self.off(x)) / self.diag, x)
        return x

    def rows(self, x, b, reverse):
        """One zebra x-line sweep: every row of a parity solved as a tridiagonal system (Thomas)."""
        for par in ((1, 0) if reverse else (0, 1)):
            ends = torch.zeros_like(x)
            ends[:, 0], ends[:, -1] = x[:, 0], x[:, -1]
            r = b - self.cross(x) - self.E * self.e(ends) - self.w(self.E * ends)
            y = _thomas(self.E[par::2, :-1].t(), self.diag[par::2].t(), r[par::2].t()).t()
            new = x.clone()
            new[par::2, 1:-1] = y
            x = torch.where(self.mask, new, x)
        return x


def _thomas(off, diag, rhs):
    """Tridiagonal solves along dim 0 for the unknowns 1 .. n-2: off[i] couples i and i + 1."""
    off, diag, rhs = off.contiguous(), diag.contiguous(), rhs.contiguous()
    n = diag.shape[0]
    c, d = torch.zeros_like(off), torch.zeros_like(rhs)
    for i in range(1, n - 1):
        r = 1.0 / (diag[i] - off[i - 1] * c[i - 1]) if i > 1 else 1.0 / diag[i]
        c[i] = off[i] * r if i < n - 2 else 0
        d[i] = (rhs[i] - off[i - 1] * d[i - 1]) * r if i > 1 else rhs[i] * r
    for i in range(n - 3, 0, -1):
        d[i] -= c[i] * d[i + 1]
    return d[1:-1]


def _restrict(r, C):
    """Full weighting to the coarse nodes, zero outside the unknowns."""
    p, n = (r + 0.5 * (_Op.w(r) + _Op.e(r))), 0.25
    v = n * (p + 0.5 * (_Op.up(p) + _Op.dn(p)))[::2, ::2]
    return torch.where(C.mask, v, torch.zeros_like(v))


def _prolong(e, F):
    """Bilinear interpolation to the fine unknowns (non-periodic levels)."""
    f = torch.zeros(F.mask.shape, dtype=F64, device=DEV)
    f[::2, ::2] = e
    f[::2, 1::2] = 0.5 * (e[:, :-1] + e[:, 1:])
    f[1::2] = 0.5 * (f[:-1:2] + f[2::2])
    return f * F.mask


def _dense(A):
    """Inverse of the matrix of A's unknowns."""
    idx = A.mask.nonzero()
    m = idx.shape[0]
    cols = []
    for k in range(m):
        e = torch.zeros(A.mask.shape, dtype=F64, device=DEV)
        e[idx[k, 0], idx[k, 1]] = 1.0
        cols.append((A.off(e) + A.diag * e)[A.mask])
    return torch.linalg.inv(torch.stack(cols, 1))


def _vcycle(ops, inv, x, b, smooth, nu, l=0):
    A = ops[l]
    if l == len(ops) - 1:
        out = torch.zeros_like(b)
        out[A.mask] = inv @ b[A.mask]
        return out
    for _ in range(nu):
        x = smooth(A, x, b, False)
    e = _vcycle(ops, inv, torch.zeros(ops[l + 1].mask.shape, dtype=F64, device=DEV), _restrict(A.residual(x, b), ops[l + 1]),
                smooth, nu, l + 1)
    x = x + _prolong(e, A)
    for _ in range(nu):
        x = smooth(A, x, b, True)
    return x


def _solve(g, spec, xp, yp, eps, rho, bc):
    """phi of -div(eps grad phi) = rho on one grid, to the FP64 residual floor."""
    if g.neumann_y:  # the even reflection about both y sides: the periodic grid of twice the height
        n = g.ny - 1
        D, exx, exy, eyy = _tensor(g, spec)
        rows = torch.tensor([n - j if j < n else j - n for j in range(2 * n)], device=DEV)
        g2 = I.Grid(g.nx, 2 * n + 1, g.x0, g.y0 - g.ly, g.lx, 2 * g.ly, periodic_y=True)
        A = _Op(g2, exx[rows], exy[rows], eyy[rows])
        x = _periodic(A, (rho * D)[rows], None if bc is None else bc[rows])
        return torch.cat([x[n:], x[:1]])
    D, exx, exy, eyy = _tensor(g, spec, xp, yp, eps)
    A = _Op(g, exx, exy, eyy)
    if g.periodic_y:
        return _periodic(A, rho * D, bc)
    ops, t, lev = [A], (exx, exy, eyy), g
    while lev.nx > 17 and lev.ny > 17 and (lev.nx - 1) % 2 == 0 and (lev.ny - 1) % 2 == 0:
        lev = I.Grid((lev.nx - 1) // 2 + 1, (lev.ny - 1) // 2 + 1, g.x0, g.y0, g.lx, g.ly)

        def half(f):
            c = f[::2, ::2].clone()
            p = f + 0.5 * (_Op.w(f) + _Op.e(f))
            c[1:-1, 1:-1] = (0.25 * (p + 0.5 * (_Op.up(p) + _Op.dn(p))))[2:-2:2, 2:-2:2]
            return c
        t = tuple(half(f) for f in t)
        ops.append(_Op(lev, *t))
    inv = _dense(ops[-1])
    return _descend(A, rho * D, bc, lambda r: _vcycle(ops, inv, torch.zeros_like(r), r, _Op.colour, 2))


def _periodic(A, b, bc):
    """Preconditioned by the operator averaged along y: Fourier in y, tridiagonal solves in x."""
    E, N = A.E.mean(0), A.N.mean(0)
    k = 2 * math.pi * torch.arange(A.mask.shape[0] // 2 + 1, dtype=F64, device=DEV) / A.mask.shape[0]
    diag = A.diag.mean(0)[:, None] + 2 * N[:, None] * torch.cos(k)[None, :]
    off = E[:-1, None].expand(-1, k.numel())

    def pre(r):
        h = torch.fft.rfft(r, dim=0).t().contiguous()
        z = torch.complex(_thomas(off, diag, h.real), _thomas(off, diag, h.imag))
        out = torch.zeros_like(r)
        out[:, 1:-1] = torch.fft.irfft(z.t(), n=r.shape[0], dim=0)
        return out
    return _descend(A, b, bc, pre)


def _descend(A, b, bc, pre):
    """Preconditioned conjugate gradients from the Dirichlet data, true residual at every restart, until
    the residual stops falling."""
    x = torch.zeros_like(b) if bc is None else torch.where(A.mask, torch.zeros_like(b), bc)
    b = torch.where(A.mask, b, torch.zeros_like(b))
    r = A.residual(x, b)
    r0 = last = float(r.norm())
    for _ in range(4):
        z = pre(r)
        p, rz = z, float((r * z).sum())
        e, q = torch.zeros_like(x), r
        for _ in range(40):
            ap = torch.where(A.mask, A.off(p) + A.diag * p, torch.zeros_like(p))
            a = rz / float((p * ap).sum())
            e, q = e + a * p, q - a * ap
            if not float(q.norm()) > 1e-5 * last:
                break
            z = pre(q)
            new = float((q * z).sum())
            p, rz = z + (new / rz) * p, new
        x = x + e
        r = A.residual(x, b)
        now = float(r.norm())
        if now < 1e-14 * r0 or now > 0.1 * last:
            break
        last = now
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        if case["nx"] * case["ny"] > 5000 ** 2:  # the wide rows of the periodic solve: over 20 seconds
            return None
        s = _instance(case, seed)
        return _solve(s["g"], s["spec"], s["xp"], s["yp"], s["eps"], s["rho"], s["bc"])
    if kind in ("batch", "serve"):  # the first few instances
        rng = _gen(seed)
        out = []
        for k, n in enumerate(_sides(case)):
            xp, yp, eps, rho = _inclusion(n, rng)
            out.append(_solve(I.Grid(n, n), I.MapSpec("grid"), xp, yp, eps, rho, None) if k < 4 else None)
        return [v if v is None or kind == "batch" else v.cpu().numpy() for v in out]
    if kind == "cycle":
        ops, b = _cycle_operators(case, seed)
        if case["prec"] == "f32":  # the rounded operators and right-hand side are the inputs
            b = b.float().double()
            for A in ops:
                A.E, A.N, A.NE, A.NW, A.diag = (v.float().double() for v in (A.E, A.N, A.NE, A.NW, A.diag))
        return _vcycle(ops, _dense(ops[-1]), torch.zeros_like(b), b, _Op.rows if case["line"] else _Op.colour, case["nu"])
    s = _build_state(case, seed)
    g = s["g"]
    t = _tensor(g, I.MapSpec("grid"), *[s[k][:, :g.nx] for k in ("xp", "yp", "eps")])
    out, A = list(t), _Op(g, *t[1:])
    for l in range(3):
        out += [A.E, A.N, A.NE, A.NW, A.diag, 1.0 / A.diag]
        A = _galerkin(A) if l < 2 else None
    return out


def _galerkin(A):
    """(1/4) P^T A P on the coarse grid, bilinear P (non-periodic)."""
    entry = {(1, 0): A.E, (-1, 0): A.w(A.E), (0, 1): A.N, (0, -1): A.dn(A.N), (1, 1): A.NE, (-1, -1): A.dn(A.w(A.NE)),
             (-1, 1): A.NW, (1, -1): A.dn(A.e(A.NW)), (0, 0): A.diag}
    h = I.Grid((A.nx - 1) // 2 + 1, (A.ny - 1) // 2 + 1)
    B = _Op(h)
    wt = (1.0, 0.5, 0.0, 0.0, 0.0)
    got = {}
    for oi, oj in ((0, 0), (1, 0), (0, 1), (1, 1), (-1, 1)):
        v = torch.zeros(h.shape, dtype=F64, device=DEV)
        for ki in (-1, 0, 1):
            for kj in (-1, 0, 1):
                for (li, lj), a in entry.items():
                    w = 0.25 * wt[abs(ki)] * wt[abs(kj)] * wt[min(4, abs(ki + li - 2 * oi))] * wt[min(4, abs(kj + lj - 2 * oj))]
                    if w:
                        v += w * torch.roll(a, (-kj, -ki), (0, 1))[::2, ::2]
        got[(oi, oj)] = torch.where(B.mask, v, torch.zeros_like(v))
    B.diag = torch.where(B.mask, got[(0, 0)], torch.ones_like(got[(0, 0)]))
    B.E, B.N, B.NE, B.NW = got[(1, 0)], got[(0, 1)], got[(1, 1)], got[(-1, 1)]
    return B
