"""Performance cases of the MinxEnt-LBM library: what a user's program has it do.

A pass is a study's unit of work through ``lbm.Lattice``: fields in, a number
of time steps, and the fields (density, velocity, totals, stream function or
populations) out.  The sizes are those of the paper's Table II studies, of the
benchmark's workloads and of the tests, plus ragged ones between them.

A case is a dict of plain values:
  kind      run      device fields in, steps, device moments and totals out
            ldas     the same with the stream function (the cavity study's stopping rule)
            readout  moments, totals and stream function of a context that has stepped
            host     host fields in, steps, host moments out
            resume   host populations in, steps, host populations out
  flow      tube (density step), vortex (Taylor-Green), cavity, sweep (cavities over 1/tau and lid speed)
  lattice, bc, rule, compute, storage   as lbm.Lattice takes them
  members, nx_lo, nx_hi, unit, ny, size_seed, spread   instances: nx in
            [nx_lo, nx_hi] (rounded to a multiple of unit), uniform (spread
            "even") or log-uniform ("log"), ny rows (0: square)
  steps     time steps of one pass
"""
import math
import random

import numpy as np
import torch

from paper_1801_03863_gb300 import lbm


def _case(name, kind, flow, lattice, bc, rule, compute, storage, members, nx_lo, nx_hi, unit, ny, steps,
          size_seed=0, spread="log"):
    return {"name": name, "kind": kind, "flow": flow, "lattice": lattice, "bc": bc, "rule": rule,
            "compute": compute, "storage": storage, "members": members, "nx_lo": nx_lo,
            "nx_hi": nx_hi, "unit": unit, "ny": ny, "steps": steps, "size_seed": size_seed,
            "spread": spread}


def listed():
    return [
        # the paper's shock tube (Table II, row ST) in its one-dimensional form: the smallest
        # lattice in use, 400 steps in which latency and launches count
        _case("tube800_f64", "run", "tube", "d1q3", "zero_gradient", "minxent4", "f64", "f64",
              1, 800, 800, 1, 1, 400),
        # the same tube as the paper runs it: D2Q9, four rows, periodic
        _case("tube2d_800x4_f64", "run", "tube", "d2q9", "periodic", "minxent4", "f64", "f64",
              1, 800, 800, 1, 4, 400),
        # stability sweep (Sec. IV.H): 120 cavities of 17 x 17 over 1/tau and lid speed, 1000 steps
        _case("sweep120_17x17_f64", "run", "sweep", "d2q9", "cavity", "minxent4", "f64", "f64",
              120, 17, 17, 1, 0, 1000),
        # accuracy study (Sec. IV.I): one 257 x 257 cavity between two checks of its stream function
        _case("ldas257_f64", "ldas", "cavity", "d2q9", "cavity", "minxent4", "f64", "f64",
              1, 257, 257, 1, 0, 500),
        # the benchmark's tube ensemble: 4096 tubes of 200 to 20000 nodes in single precision
        _case("tubes4096_f32", "run", "tube", "d1q3", "zero_gradient", "minxent4", "f32", "f32",
              4096, 200, 20000, 1, 1, 100, size_seed=1),
        # Taylor-Green vortex, an ordinary single lattice
        _case("vortex512_f32", "run", "vortex", "d2q9", "periodic", "minxent4", "f32", "f32",
              1, 512, 512, 1, 0, 200),
        # one large cavity with 16-bit storage
        _case("cavity2048_f16", "run", "cavity", "d2q9", "cavity", "minxent4", "f32", "f16",
              1, 2048, 2048, 1, 0, 100),
        # the headline: 64 uneven cavities, 16-bit storage, totals after every 100 steps
        _case("cavities64_f16", "run", "cavity", "d2q9", "cavity", "minxent4", "f32", "f16",
              64, 64, 1024, 64, 0, 100, spread="even"),
        # ragged ensemble with one of the comparison rules and single-precision storage
        _case("ragged48_mrt_f32", "run", "cavity", "d2q9", "cavity", "mrt", "f32", "f32",
              48, 50, 1100, 1, 0, 100, size_seed=5),
        # a study driven from host arrays, as a script with numpy fields runs it
        _case("host16_minxent2_bf16", "host", "cavity", "d2q9", "cavity", "minxent2", "f32", "bf16",
              16, 90, 700, 1, 0, 200, size_seed=3),
        # a run picked up from saved populations and saved again: zero-gradient ends, odd sizes
        _case("resume1001x333_trt_f32", "resume", "vortex", "d2q9", "zero_gradient", "trt", "f32",
              "f32", 1, 1001, 1001, 1, 333, 60),
        # reading out an ensemble between bursts of steps: moments, totals, stream function
        _case("readout64_f16", "readout", "cavity", "d2q9", "cavity", "minxent4", "f32", "f16",
              64, 64, 1024, 1, 0, 20, size_seed=7),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds with sizes over their whole range."""
    flow = rng.choice(["tube", "tube", "tubes", "sweep", "cavity", "cavity", "cavities", "cavities", "vortex"])
    compute = "f64" if rng.random() < (0.6 if flow in ("tube", "sweep") else 0.2) else "f32"
    storage = "f64" if compute == "f64" else rng.choice(["f32", "f16", "f16", "bf16"])
    rule = rng.choice(["minxent4", "minxent4", "minxent4", "minxent2", "srt", "mrt", "trt"])
    size_seed = rng.randrange(1 << 20)
    kind = "run"
    if flow in ("tube", "tubes"):
        members = 1 if flow == "tube" else _log_int(rng, 8, 4096)
        if members == 1 and rng.random() < 0.4:  # two-dimensional form
            nx, ny, lattice, bc = _log_int(rng, 100, 2000), rng.randint(2, 9), "d2q9", "periodic"
        else:
            nx, ny, lattice = _log_int(rng, 50, 20000), 1, "d1q3"
            bc = rng.choice(["zero_gradient", "zero_gradient", "periodic"])
        if lattice == "d1q3":
            rule = "minxent4"
        storage = "f64" if compute == "f64" else "f32"
        c = _case("", "run", "tube", lattice, bc, rule, compute, storage, members,
                  nx if members == 1 else 200, nx if members == 1 else max(nx, 400), 1, ny,
                  rng.randint(40, 400), size_seed)
    elif flow == "sweep":
        side = rng.choice([17, 17, 21, 33])
        rule = "minxent4"
        if compute == "f32":
            storage = "f32"
        c = _case("", "run", "sweep", "d2q9", "cavity", rule, compute, storage,
                  _log_int(rng, 6, 160), side, side, 1, 0, rng.randint(100, 1000), size_seed)
    elif flow == "vortex":
        nx, ny = _log_int(rng, 64, 1500), _log_int(rng, 64, 1500)
        kind = rng.choice(["run", "run", "resume"])
        bc = "periodic" if kind == "run" else rng.choice(["periodic", "zero_gradient"])
        c = _case("", kind, "vortex", "d2q9", bc, rule, compute, storage, 1, nx, nx, 1, ny,
                  rng.randint(20, 200), size_seed)
    elif flow == "cavity":
        nx = _log_int(rng, 33, 2048)
        kind = rng.choice(["run", "run", "ldas", "host"])
        c = _case("", kind, "cavity", "d2q9", "cavity", rule, compute, storage, 1, nx, nx, 1, 0,
                  rng.randint(20, 200), size_seed)
    else:
        kind = rng.choice(["run", "run", "readout", "host"])
        c = _case("", kind, "cavity", "d2q9", "cavity", rule, compute, storage,
                  _log_int(rng, 4, 72), 40, _log_int(rng, 200, 1024), rng.choice([1, 1, 8, 64]), 0,
                  rng.randint(20, 100), size_seed, rng.choice(["log", "even"]))
        c["nx_lo"] = max(c["nx_lo"], c["unit"])
    del c["name"]
    if kind in ("ldas", "readout") and storage == "bf16":
        c["storage"] = "f16"  # eight bits do not resolve a stream function
    # no larger than the largest listed cases: about 25 ms of steps, and host
    # arrays of a few million nodes
    rate = {"f64": 1.0e9}.get(compute, 80.0e9)
    while c["members"] > 4 and _nodes(c) > (3.0e6 if c["kind"] in ("host", "resume") else 1.5e7):
        c["members"] = c["members"] * 3 // 4
    c["steps"] = max(4, min(c["steps"], int(0.025 * rate / _nodes(c))))
    return c


# ----------------------------------------------------------------------------
# Inputs.
# ----------------------------------------------------------------------------
def _dims(case):
    rng = random.Random(case["size_seed"])
    out = []
    for _ in range(case["members"]):
        n = rng.randint(case["nx_lo"], case["nx_hi"]) if case["spread"] == "even" else \
            _log_int(rng, case["nx_lo"], case["nx_hi"])
        n = max(case["unit"], int(round(n / case["unit"])) * case["unit"])
        out.append((n, case["ny"] if case["ny"] else n))
    return out


def _nodes(case):
    return sum(a * b for a, b in _dims(case))


def _inputs(case, seed):
    """Instance sizes, viscosities, lid speeds, reference density and the
    initial fields (device FP64, instances concatenated)."""
    dims = _dims(case)
    rng = random.Random(1000003 * int(seed) + 17)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    n = len(dims)
    total = sum(a * b for a, b in dims)
    rho0, lids = 1.0, [0.0] * n
    noise = 1e-6 * (2.0 * torch.rand(total, generator=gen, device="cuda", dtype=torch.float64) - 1.0)
    ux = torch.zeros(total, device="cuda", dtype=torch.float64)
    uy = torch.zeros(total, device="cuda", dtype=torch.float64)
    if case["flow"] == "tube":
        # Table II: density step, at rest but for a shear wave across the tube
        # in the two-dimensional form (nearly inviscid, as the paper's, so
        # that the wave lives on); viscosities of the others from the upper part of
        # the tube ensemble's range, where every run stays stable
        lo, hi = (1e-4, 5e-4) if case["ny"] > 1 else (2e-3, 2e-2)
        nus = [math.exp(rng.uniform(math.log(lo), math.log(hi))) for _ in dims]
        ratio = torch.tensor([rng.uniform(1.5, 3.0) for _ in dims], device="cuda", dtype=torch.float64)
        sizes = torch.tensor([a * b for a, b in dims], device="cuda")
        inst = torch.repeat_interleave(torch.arange(n, device="cuda"), sizes)
        start = torch.cumsum(sizes, 0) - sizes
        widths = torch.tensor([a for a, _ in dims], device="cuda")
        k = torch.arange(total, device="cuda") - start[inst]
        x = k % widths[inst]
        if case["ny"] > 1:
            wave = 2.0 * math.pi * (rng.random() + 8.0 * x.double() / case["nx_lo"])
            uy = (0.02 * torch.cos(wave)).contiguous()
        rho = noise + torch.where(x < widths[inst] // 2, ratio[inst], torch.ones_like(noise))
    elif case["flow"] == "vortex":
        (nx, ny), = dims
        u0 = rng.uniform(0.02, 0.05)
        nus = [math.exp(rng.uniform(math.log(1e-3), math.log(1e-2)))]
        x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :] * (2.0 * math.pi / nx)
        y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None] * (2.0 * math.pi / ny)
        ux = (-u0 * torch.cos(x) * torch.sin(y)).reshape(-1).contiguous()
        uy = (u0 * torch.sin(x) * torch.cos(y)).reshape(-1).contiguous()
        rho = (1.0 - 0.75 * u0 * u0 * (torch.cos(2 * x) + torch.cos(2 * y))).reshape(-1) + noise
    elif case["flow"] == "sweep":
        rho0 = 2.7
        lids = [rng.uniform(0.05, 0.25) for _ in dims]
        nus = [(1.0 / rng.uniform(1.0, 1.9) - 0.5) / 3.0 for _ in dims]
        rho = rho0 + noise
    else:
        rho0 = 2.7 if case["kind"] == "ldas" else 1.0
        lids = [rng.uniform(0.05, 0.1) for _ in dims]
        nus = [u * nx / math.exp(rng.uniform(math.log(100.0), math.log(2000.0)))
               for u, (nx, _) in zip(lids, dims)]
        rho = rho0 + noise
    return dims, nus, lids, rho0, rho.contiguous(), ux, uy


def prepare(case, seed):
    """The context a program keeps, and its fields; results go to buffers of its own."""
    dims, nus, lids, rho0, rho, ux, uy = _inputs(case, seed)
    lat = lbm.Lattice(case["lattice"], dims, nus, case["bc"],
                      u_lid=lids if case["bc"] == "cavity" else None, compute=case["compute"],
                      storage=case["storage"], collision=case["rule"], rho0=rho0,
                      stream=torch.cuda.current_stream())
    two = lat.q == 9
    st = {"kind": case["kind"], "steps": case["steps"], "lat": lat, "two": two}
    if case["kind"] == "host":
        st["host"] = [t.cpu().numpy() for t in ((rho, ux, uy) if two else (rho, ux))]
        return st
    if case["kind"] == "resume":
        # populations near equilibrium, as a saved run has them
        f = _equilibrium(rho, ux, uy if two else None)
        k, parts = 0, []
        for nx, ny in dims:
            parts += [fa[k:k + nx * ny] for fa in f]
            k += nx * ny
        st["host"] = torch.cat(parts).cpu().numpy()
        return st
    st["in"] = (rho, ux, uy) if two else (rho, ux)
    st["out"] = [torch.empty_like(rho) for _ in st["in"]]
    st["totals"] = torch.empty(3 * len(dims), device="cuda", dtype=torch.float64)
    st["psi"] = torch.empty_like(rho) if case["kind"] in ("ldas", "readout") else None
    if case["kind"] == "readout":
        lat.init_device(*st["in"])
        lat.step(case["steps"])
        torch.cuda.synchronize()
    return st


def run(state):
    lat = state["lat"]
    if state["kind"] == "host":
        lat.init(*state["host"])
        lat.step(state["steps"])
        rho, ux, uy = lat.moments(allow_unstable=True)
        return {"rho": rho, "ux": ux, "uy": uy} if state["two"] else {"rho": rho, "ux": ux}
    if state["kind"] == "resume":
        lat.set_populations(state["host"])
        lat.step(state["steps"])
        return {"f": lat.populations()}
    if state["kind"] != "readout":
        lat.init_device(*state["in"])
        lat.step(state["steps"])
    lat.conservation_device(state["totals"])
    lat.moments_device(*state["out"])
    out = dict(zip(("rho", "ux", "uy"), state["out"]), totals=state["totals"])
    if state["psi"] is not None:
        lat.stream_function_device(state["psi"])
        out["psi"] = state["psi"]
    return out


def work(case):
    """Fields in and out once, and the arithmetic of every lattice update."""
    n, two = _nodes(case), case["lattice"] == "d2q9"
    fields = 8 * (3 if two else 2) * n
    es = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}[case["storage"]]
    per = {"minxent4": 400, "minxent2": 280, "srt": 110, "mrt": 110, "trt": 110}[case["rule"]]
    flops = n * case["steps"] * (per if two else 40)
    if case["kind"] == "readout":
        return {"bytes": 9 * es * n + fields + 8 * n, "flops": 30 * n}
    if case["kind"] == "resume":
        return {"bytes": 2 * 72 * n, "flops": flops}
    return {"bytes": 2 * fields + (8 * n if case["kind"] == "ldas" else 0), "flops": flops}


# ----------------------------------------------------------------------------
# The same in plain 64-bit torch, written from the paper: Eq. (2) with the
# boundary rules of Sec. IV.F, Eqs. (bgkcollision), (mrtcollision) and the
# single Newton step of Sec. IV.C-E.
# ----------------------------------------------------------------------------
_VX9, _VY9 = [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1]
_W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
_OPP9 = [0, 3, 4, 1, 2, 7, 8, 5, 6]
_T = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], _VX9,
      [0, -2, 0, 2, 0, 1, -1, -1, 1], _VY9, [0, 0, -2, 0, 2, 1, 1, -1, -1],
      [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]
_D = [sum(v * v for v in row) for row in _T]  # T T^t = diag(_D)


def _equilibrium(rho, ux, uy):
    if uy is None:
        vx, vy, w = [0, 1, -1], [0, 0, 0], [2 / 3, 1 / 6, 1 / 6]
        uy = torch.zeros_like(ux)
    else:
        vx, vy, w = _VX9, _VY9, _W9
    b = 1.5 * (ux * ux + uy * uy)
    out = []
    for a in range(len(w)):
        vu = vx[a] * ux + vy[a] * uy
        out.append(w[a] * rho * (1.0 + 3.0 * vu + 4.5 * vu * vu - b))
    return out


def _moments(f):
    vx, vy = (_VX9, _VY9) if len(f) == 9 else ([0, 1, -1], [0, 0, 0])
    rho = sum(f[1:], f[0])
    jx = sum(v * x for v, x in zip(vx, f) if v)
    jy = sum(v * x for v, x in zip(vy, f) if v) if len(f) == 9 else None
    return rho, jx / rho, None if jy is None else jy / rho


def _rows(coef, v):
    return sum(c * x for c, x in zip(coef, v) if c)


def _collide(f, rule, om, om2):
    rho, ux, uy = _moments(f)
    feq = _equilibrium(rho, ux, uy)
    if len(f) == 3 or rule == "srt":
        return [x + om * (e - x) for x, e in zip(f, feq)]
    if rule in ("mrt", "trt"):
        rates = [0, om if rule == "trt" else 1.64, om if rule == "trt" else 1.54, 0, om2, 0, om2, om, om]
        post = list(f)
        for k in (1, 2, 4, 6, 7, 8):
            step = rates[k] * (_rows(_T[k], feq) - _rows(_T[k], f)) / _D[k]
            post = [x + c * step if c else x for x, c in zip(post, _T[k])]
        return post
    p = [e / rho for e in feq]
    for k, rate in [(7, om), (8, om)] + ([(4, om2), (6, om2)] if rule == "minxent2" else []):
        step = (1.0 - rate) * (_rows(_T[k], f) - _rows(_T[k], feq)) / (rho * _D[k])
        p = [x + c * step if c else x for x, c in zip(p, _T[k])]
    free = (1, 2, 4, 6) if rule == "minxent4" else (1, 2)
    good = torch.ones_like(rho, dtype=torch.bool)
    for x in p:
        good &= x > 0
    lg = [torch.log(x / w) for x, w in zip(p, _W9)]
    inv = [1.0 / x for x in p]
    m = len(free)
    b = [_rows(_T[k], lg) for k in free]
    A = [[_rows([s * t for s, t in zip(_T[j], _T[k])], inv) for k in free] for j in free]
    for i in range(m):  # symmetric positive definite: elimination without pivoting
        for r in range(i + 1, m):
            q = A[r][i] / A[i][i]
            for c in range(i, m):
                A[r][c] = A[r][c] - q * A[i][c]
            b[r] = b[r] - q * b[i]
    s = [None] * m
    for i in reversed(range(m)):
        s[i] = (b[i] - sum(A[i][c] * s[c] for c in range(i + 1, m))) / A[i][i]
    s = [torch.where(good, x, torch.zeros_like(x)) for x in s]
    return [rho * (x - sum(_T[k][a] * y for k, y in zip(free, s))) for a, x in enumerate(p)]


def exact(case, seed):
    dims, nus, lids, rho0, rho, ux, uy = _inputs(case, seed)
    two = case["lattice"] == "d2q9"
    if not two:
        uy = None
    vx, vy, w = (_VX9, _VY9, _W9) if two else ([0, 1, -1], [0, 0, 0], [2 / 3, 1 / 6, 1 / 6])
    dev, bc = "cuda", case["bc"]
    sizes = torch.tensor([a * b for a, b in dims], device=dev)
    inst = torch.repeat_interleave(torch.arange(len(dims), device=dev), sizes)
    start = (torch.cumsum(sizes, 0) - sizes)[inst]
    nx = torch.tensor([a for a, _ in dims], device=dev)[inst]
    ny = torch.tensor([b for _, b in dims], device=dev)[inst]
    k = torch.arange(rho.numel(), device=dev) - start
    x, y = k % nx, k // nx
    src, ok = [], []
    for a in range(len(w)):
        sx, sy = x - vx[a], y - vy[a]
        if bc == "cavity":
            inside = (sx >= 0) & (sx < nx) & (sy >= 0) & (sy < ny)
            sx, sy = torch.where(inside, sx, x), torch.where(inside, sy, y)
            ok.append(inside)
        else:
            sx = sx % nx if bc == "periodic" else torch.minimum(torch.clamp(sx, min=0), nx - 1)
            sy = sy % ny
        src.append(start + sy * nx + sx)
    wall = (x == 0) | (x == nx - 1) | (y == 0)
    lid = ~wall & (y == ny - 1)
    del sx, sy, k
    nu = torch.tensor(nus, device=dev, dtype=torch.float64)
    tau = 3.0 * nu + 0.5
    om, om2 = (1.0 / tau)[inst], ((2.0 * tau - 1.0) / (8.0 * tau - 1.0))[inst]
    u = torch.tensor(lids, device=dev, dtype=torch.float64)[inst]
    flid = [torch.where(lid, e, 0.0) for e in _equilibrium(torch.full_like(u, rho0), u, torch.zeros_like(u))] \
        if bc == "cavity" else None
    f = _equilibrium(rho, ux, uy)
    for _ in range(case["steps"]):
        post = _collide(f, case["rule"], om, om2)
        if bc == "cavity":
            post = [torch.where(wall, f[_OPP9[a]], torch.where(lid, flid[a], post[a])) for a in range(9)]
            f = [torch.where(ok[a], post[a][src[a]], torch.full_like(rho, w[a] * rho0)) for a in range(9)]
        else:
            f = [post[a][src[a]] for a in range(len(w))]
    if case["kind"] == "resume":
        kk, parts = 0, []
        for a, b in dims:
            parts += [fa[kk:kk + a * b] for fa in f]
            kk += a * b
        return {"f": torch.cat(parts)}
    r, vxm, vym = _moments(f)
    out = {"rho": r, "ux": vxm}
    if two:
        out["uy"] = vym
    if case["kind"] == "host":
        return out
    sums = [torch.zeros(len(dims), device=dev, dtype=torch.float64).index_add_(0, inst, q)
            for q in (r, r * vxm, r * vym if two else torch.zeros_like(r))]
    out["totals"] = torch.stack(sums, 1).reshape(-1)
    if case["kind"] in ("ldas", "readout"):
        # composite Simpson rule along each row, trapezoid on a last odd interval
        psi, at = [], 0
        for a, b in dims:
            v = vym[at:at + a * b].reshape(b, a)
            p = torch.zeros_like(v)
            pairs = (v[:, 0:-2:2] + 4.0 * v[:, 1:-1:2] + v[:, 2::2]) / 3.0
            even = torch.cumsum(pairs, 1)
            p[:, 2::2] = -even
            base = torch.cat([torch.zeros_like(v[:, :1]), even], 1)
            odd = 0.5 * (v[:, 0:-1:2] + v[:, 1::2])
            p[:, 1::2] = -(base[:, :odd.shape[1]] + odd)
            psi.append(p.reshape(-1))
            at += a * b
        out["psi"] = torch.cat(psi)
    return out
