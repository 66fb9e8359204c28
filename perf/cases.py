"""The solver work that is timed: what users of this package have it do, through its public calls.

A case is one of six kinds:

  tube    a shock tube a few rows high (Sec. 5.1), periodic in y, outflow in x
  quad    a two-dimensional four-quadrant problem, outflow on every side or periodic
  dmr     the double Mach reflection (Sec. 5.2.2): Dirichlet sides, a wall, segments that move
  steady  the regular reflection (Sec. 5.2) in the canonical-order FP64 precision
  batch   a set of resident serving tubes of mixed length advanced together (fdlbm_batch_*)
  vn      the von Neumann sweep of Sec. 4: spectra of the 33 x 33 amplification matrix

For the solves a pass is a whole short solve on the device: the initial condition from the user's
arrays (fdlbm_set_macro_device, or fdlbm_set_macro from host arrays), `steps` time steps, and the
macros read out. Real runs take thousands of steps, so `steps` is large enough that the steps are
most of a pass. A batch has no initial condition inside its pass: a server's members stay resident
and are advanced round by round, so a pass advances them by `steps` and reads every member's macros.

Initial fields carry a smooth perturbation of a few per cent: after its first steps a real flow has
no two equal nodes, and no exactly constant region. Shock strengths stay where an FP64 solve
determines its result to 1e-9 (the conditioning sum|f|/n grows fast with the Mach number); the
Mach-20 reflection runs in the precision whose operation order is fixed.
"""
import math

import numpy as np
import torch

from paper_0801_4169_gb300 import fdlbm as F
from paper_0801_4169_gb300 import workloads as W

PREC = {"fp64": F.FDLBM_FP64, "fp32": F.FDLBM_FP32_STORE, "fneq32": F.FDLBM_FNEQ32, "dw": F.FDLBM_FP32_STORE_DW,
        "strict": F.FDLBM_FP64_STRICT}
F32_STATE = ("fp32", "dw")  # state buffers and results are FP32 numbers
DEVICE = "cuda"


def listed():
    return [
        # the tube of Sec. 5.1 as a user studies it: 1600 sites, a step is a few microseconds
        {"name": "sod_400x4_fp64", "kind": "tube", "nx": 400, "ny": 4, "prec": "fp64", "Ms": 0.0, "steps": 64,
         "r": 1.0, "flags": 0, "host": False},
        # a strong-shock tube, called with host arrays as from a script
        {"name": "shock_4000x4_fp64_host", "kind": "tube", "nx": 4000, "ny": 4, "prec": "fp64", "Ms": 5.0,
         "steps": 50, "r": 1.0, "flags": 0, "host": True},
        # the double Mach reflection at the paper's grid: walls, Dirichlet sides, moving segments
        {"name": "dmr_500x200_fp64", "kind": "dmr", "nx": 500, "ny": 200, "steps": 20},
        # an ordinary two-dimensional study, odd and ragged, tau = 4 dt
        {"name": "quad_1023x777_fp64", "kind": "quad", "nx": 1023, "ny": 777, "prec": "fp64", "steps": 8, "r": 0.25,
         "periodic": False},
        # a large FP64 solve
        {"name": "quad_2048x2048_fp64", "kind": "quad", "nx": 2048, "ny": 2048, "prec": "fp64", "steps": 6, "r": 1.0,
         "periodic": False},
        # the headline grid in FP32 storage
        {"name": "quad_4096x4096_fp32", "kind": "quad", "nx": 4096, "ny": 4096, "prec": "fp32", "steps": 10, "r": 1.0,
         "periodic": False},
        # a parameter study in FP32 storage: a ragged middle size
        {"name": "quad_517x333_fp32", "kind": "quad", "nx": 517, "ny": 333, "prec": "fp32", "steps": 24, "r": 1.0,
         "periodic": True},
        # the double-word option on a large grid
        {"name": "quad_2048x2048_dw", "kind": "quad", "nx": 2048, "ny": 2048, "prec": "dw", "steps": 12, "r": 1.0,
         "periodic": False},
        # departure-from-equilibrium storage: FP64-class results in less memory
        {"name": "quad_1000x1000_fneq32", "kind": "quad", "nx": 1000, "ny": 1000, "prec": "fneq32", "steps": 8,
         "r": 1.0, "periodic": False},
        # the Mach-20 reflection checked in the canonical operation order
        {"name": "reflection_300x75_strict", "kind": "steady", "nx": 300, "ny": 75, "steps": 8},
        # continuous serving: resident tubes of the request stream's sizes, one round's slice
        {"name": "serve_32_tubes_fp64", "kind": "batch", "members": 32, "lo": 256, "hi": 16384, "prec": "fp64",
         "steps": 24},
        # the Sec. 4 sweep: 22 curves over the wave number
        {"name": "vn_sec4_256", "kind": "vn", "nk": 256},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tube", "tube", "quad", "quad", "quad", "dmr", "steady", "batch", "vn"])
    if kind == "tube":
        prec = rng.choice(["fp64", "fp64", "fp32", "fneq32", "dw"])
        return {"kind": kind, "nx": _log(rng, 200, 16384), "ny": rng.choice([1, 3, 4, 4, 4, 5]), "prec": prec,
                "Ms": rng.choice([0.0, rng.uniform(2.0, 6.0 if prec in ("fp64", "fneq32") else 3.0)]),
                "steps": _log(rng, 16, 90), "r": rng.choice([1.0, 0.1]), "flags": rng.choice([0, 0, 0, W._NO_DISP]),
                "host": rng.random() < 0.3}
    if kind == "quad":
        prec = rng.choice(["fp64", "fp64", "fp32", "fp32", "dw", "fneq32"])
        sites = _log(rng, 8000, 4.2e6 if prec in ("fp64", "fneq32") else 1.6e7)
        nx = max(64, int(math.sqrt(sites) * math.exp(rng.uniform(-0.7, 0.7))))
        return {"kind": kind, "nx": nx, "ny": max(32, sites // nx), "prec": prec,
                "steps": max(2, min(40, int(2e7 / sites))), "r": rng.choice([1.0, 1.0, 0.25]),
                "periodic": rng.random() < 0.4}
    if kind == "dmr":
        nx = _log(rng, 150, 1200)
        return {"kind": kind, "nx": nx, "ny": int(nx * rng.uniform(0.3, 0.5)), "steps": rng.randint(10, 30)}
    if kind == "steady":
        ny = _log(rng, 24, 150)
        return {"kind": kind, "nx": 4 * ny + rng.randint(0, 7), "ny": ny, "steps": rng.randint(4, 10)}
    if kind == "batch":
        return {"kind": kind, "members": rng.randint(4, 60), "lo": 256, "hi": _log(rng, 1024, 16384),
                "prec": rng.choice(["fp64", "fp64", "fneq32"]), "steps": rng.randint(8, 32)}
    return {"kind": "vn", "nk": _log(rng, 8, 250)}


# ---------------------------------------------------------------------------------------------
# inputs


def _perturb(shape, dx, rng, amp, count=3):
    """A smooth field of `count` waves along each axis with random phases, of size amp."""
    ny, nx = shape
    x = torch.arange(nx, dtype=torch.float64, device=DEVICE)[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=DEVICE)[:, None]
    out = torch.zeros(shape, dtype=torch.float64, device=DEVICE)
    for _ in range(count):
        kx = 2 * math.pi * int(rng.integers(1, 6)) / nx
        ky = 2 * math.pi * int(rng.integers(0, 3)) / ny
        out += (amp / count) * torch.sin(kx * x + ky * y + float(rng.uniform(0, 2 * math.pi)))
    return out


def _full(shape, value):
    return torch.full(shape, float(value), dtype=torch.float64, device=DEVICE)


def _problem(case, seed):
    """(parameters, device fields) of a solve; parameters as keyword arguments of fdlbm.Solver plus segments."""
    rng = np.random.Generator(np.random.PCG64(seed))
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    shape = (ny, nx)
    seg, bstate = (), np.zeros((4, 4))
    flags, prec = case.get("flags", 0), case.get("prec", "fp64")
    if kind == "tube":
        dx, dt, lam = 1e-3, 1e-5, 2.0
        bc = (W.OUTFLOW, W.OUTFLOW, W.PERIODIC, W.PERIODIC)
        if case["Ms"]:
            c1 = math.sqrt(W.GAMMA * 0.5)
            u1 = -max(0.0, case["Ms"] - 2.0) * c1
            rho2, u2, T2, _ = W.rh_moving_shock(case["Ms"], 1.0, 0.5, u1)
            left, right, x0 = (rho2, u2, 0.0, T2), (1.0, u1, 0.0, 0.5), rng.uniform(0.1, 0.3)
        else:
            left, right, x0 = (1.0, 0.0, 0.0, 1.0), (rng.uniform(0.12, 0.3), 0.0, 0.0, 0.8), rng.uniform(0.4, 0.6)
        split = torch.arange(nx, device=DEVICE)[None, :].expand(shape) < x0 * nx
        f = [torch.where(split, _full(shape, a), _full(shape, b)) for a, b in zip(left, right)]
    elif kind == "quad":
        dx, dt, lam = 2.5e-4, 2.5e-6, 3.0
        bc = (W.PERIODIC,) * 4 if case["periodic"] else (W.OUTFLOW,) * 4
        st = W.riemann4q(n=2, seed=seed).meta["states"]
        ix = (torch.arange(nx, device=DEVICE) >= nx // 2)[None, :]
        iy = (torch.arange(ny, device=DEVICE) >= ny // 2)[:, None]
        f = []
        for i in range(4):
            lo = torch.where(ix, _full((1, nx), st[1][i]), _full((1, nx), st[0][i]))
            hi = torch.where(ix, _full((1, nx), st[3][i]), _full((1, nx), st[2][i]))
            f.append(torch.where(iy, hi, lo).contiguous())
    elif kind == "dmr":
        w = W.dmr(Ms=6.0, nx=nx, ny=ny)
        dx, dt, lam, bc, bstate, seg = w.dx, w.dt, w.lam, w.bc, w.bstate, w.meta["segments"]
        f = [torch.from_numpy(np.array(a)).to(DEVICE) for a in w.macros()]
    else:
        w = W.reflection(nx=nx, ny=ny)
        dx, dt, lam, bc, bstate, prec = w.dx, w.dt, w.lam, w.bc, w.bstate, "strict"
        f = [torch.from_numpy(np.array(a)).to(DEVICE) for a in w.macros()]
    amp = 0.005 if kind == "steady" else 0.03
    f[0] = f[0] * (1.0 + _perturb(shape, dx, rng, amp))
    f[1] = f[1] + _perturb(shape, dx, rng, amp)
    f[2] = f[2] + _perturb(shape, dx, rng, amp)
    f[3] = f[3] * (1.0 + _perturb(shape, dx, rng, amp))
    par = dict(nx=nx, ny=ny, dx=dx, dy=dx, dt=dt, tau=dt / case.get("r", 1.0), lam=lam, bc=bc, prec=PREC[prec],
               flags=flags, bstate=bstate)
    return par, seg, [a.contiguous() for a in f]


def _state_view(s, prec):
    """Interior of the two state buffers [33, ny, nx] in the storage type, from the caller's torch memory."""
    pitch, rows = (s.nx + 4 + 31) // 32 * 32, s.ny + 4
    ty, es = (torch.float32, 4) if prec in F32_STATE else (torch.float64, 8)
    n = 33 * pitch * rows * es
    fbytes = (n + 255) // 256 * 256
    views = []
    for b in range(2):
        at = s.mem_offset + b * fbytes
        views.append(s._mem[at:at + n].view(ty).view(33, rows, pitch)[:, 2:2 + s.ny, 2:2 + s.nx])
    return views


def _batch_members(case, seed):
    sizes = np.random.Generator(np.random.PCG64(case["members"])).integers(case["lo"], case["hi"] + 1, case["members"])
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for i in range(case["members"]):
        nx = int(sizes[i]) if i else case["hi"]
        out.append(({"kind": "tube", "nx": nx, "ny": 4, "prec": case["prec"], "Ms": float(rng.uniform(2.0, 5.0)),
                     "r": 1.0, "flags": 0}, int(rng.integers(1 << 30))))
    return out


def _vn_rows(case, seed):
    """The Sec. 4 sweep around its states: (n, u1, u2, T, xi_x, xi_y, lambda, flags) per row."""
    rng = np.random.Generator(np.random.PCG64(seed))
    rows, _, _ = W.vn_sec4_cases(case["nk"])
    rows[:, 0] *= rng.uniform(0.9, 1.1, len(rows))
    rows[:, 3] *= rng.uniform(0.98, 1.02, len(rows))
    return rows


def prepare(case, seed):
    stream = torch.cuda.current_stream()
    if case["kind"] == "vn":
        rows = _vn_rows(case, seed)
        c = F.vn_cases(rows[:, :4], rows[:, 4], rows[:, 5], rows[:, 6], rows[:, 7].astype(np.int32))
        n = len(c)
        return {"kind": "vn", "n": n, "cases": torch.from_numpy(c.view(np.uint8).copy()).to(DEVICE),
                "max_abs": torch.empty(n, dtype=torch.float64, device=DEVICE),
                "G": torch.empty((n, 33, 33, 2), dtype=torch.float64, device=DEVICE),
                "status": torch.empty(n, dtype=torch.int32, device=DEVICE), "stream": stream}
    if case["kind"] == "batch":
        b = F.fdlbm_batch_create(stream)
        solvers, at, spans = [], 0, []
        for sub, s in _batch_members(case, seed):
            par, _, f = _problem(sub, s)
            sv = F.Solver(stream=stream, **par)
            F.fdlbm_set_macro_device(sv.h, *f)
            F.fdlbm_batch_add(b, sv.h)
            solvers.append(sv)
            spans.append((at, sub["nx"] * 4))
            at += sub["nx"] * 4
        return {"kind": "batch", "b": _Batch(b, solvers), "spans": spans, "steps": case["steps"],
                "out": torch.empty((4, at), dtype=torch.float64, device=DEVICE)}
    par, seg, f = _problem(case, seed)
    s = F.Solver(stream=stream, **par)
    for side, c0, speed, lower, st in seg:
        F.fdlbm_set_boundary_segment(s.h, side, c0, speed, lower, *st)
    prec = "strict" if case["kind"] == "steady" else case.get("prec", "fp64")
    state = {"kind": "solve", "s": s, "steps": case["steps"], "host": case.get("host", False), "prec": prec,
             "f": f, "out": torch.empty((4, case["ny"], case["nx"]), dtype=torch.float64, device=DEVICE)}
    if prec in F32_STATE:
        state["out32"] = torch.empty((4, case["ny"], case["nx"]), dtype=torch.float32, device=DEVICE)
    if prec != "fneq32":
        state["view"] = _state_view(s, prec)
    if state["host"]:
        state["f"] = [a.cpu().numpy() for a in f]
    return state


class _Batch:
    """A batch and its members, taken apart in the order the library asks for."""

    def __init__(self, b, solvers):
        self.b, self.solvers = b, solvers

    def __del__(self):
        try:
            F.fdlbm_batch_destroy(self.b)
            for s in self.solvers:
                s.close()
        except Exception:
            pass


# ---------------------------------------------------------------------------------------------
# one pass


def run(state):
    if state["kind"] == "vn":
        F.fdlbm_vn_spectrum(state["cases"], state["n"], *W.VN_SEC4_GRID, state["max_abs"], None, state["G"],
                            state["status"], state["stream"])
        return {"max_abs": state["max_abs"], "G": state["G"], "status": state["status"]}
    if state["kind"] == "batch":
        out = state["out"]
        F.fdlbm_batch_step(state["b"].b, state["steps"])
        for sv, (at, n) in zip(state["b"].solvers, state["spans"]):
            F.fdlbm_get_macro_device(sv.h, *[out[i, at:at + n] for i in range(4)])
        return {"macros": out}
    s = state["s"]
    if state["host"]:
        s.set_macro(*state["f"])
        s.step(state["steps"])
        m = s.get_macro()
        if state["prec"] in F32_STATE:
            m = [a.astype(np.float32) for a in m]
    else:
        F.fdlbm_set_macro_device(s.h, *state["f"])
        s.step(state["steps"])
        out = state["out"]
        F.fdlbm_get_macro_device(s.h, out[0], out[1], out[2], out[3])
        m = out
        if state["prec"] in F32_STATE:  # an FP32 state's macros are kept as FP32 numbers
            m = state["out32"].copy_(out)
    res = {"rho": m[0], "u": m[1], "v": m[2], "T": m[3]}
    if "view" in state:
        res["f"] = state["view"][F.fdlbm_current_buffer(s.h)]
    return res


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without

# One site update: 33 values read and written; the moments (about 130 operations), the equilibrium
# (about 350) and Eq. 17 with nine points for each diagonal and seven for each axis direction (about 600).
SITE_FLOPS = 1080.0


def work(case):
    if case["kind"] == "vn":
        n = 22 * case["nk"]
        # Hessenberg reduction and shifted QR of a complex matrix of order 33: about 18 n^3 complex
        # multiply-adds (8 operations each), each carried in twice the working precision (about 20)
        return {"bytes": n * (64.0 + 8 + 4 + 2178 * 8), "flops": n * 18.0 * 33 ** 3 * 8 * 20}
    if case["kind"] == "batch":
        sites = 4.0 * sum(m["nx"] for m, _ in _batch_members(case, 0))
        value = 8 if case["prec"] == "fp64" else 4 + 4 * 8 / 33.0
        return {"bytes": sites * (case["steps"] * 66 * value + 32), "flops": sites * case["steps"] * SITE_FLOPS}
    sites = float(case["nx"]) * case["ny"]
    prec = case.get("prec", "fp64")
    value = 4 if prec in F32_STATE else 4 + 4 * 8 / 33.0 if prec == "fneq32" else 8
    return {"bytes": sites * (case["steps"] * 66 * value + 64), "flops": sites * case["steps"] * SITE_FLOPS}


# ---------------------------------------------------------------------------------------------
# the same in plain 64-bit torch, from the equations

_SPEED = (1.0, 1.92, 2.99, 4.49)
_S = math.sqrt(0.5)
_DIR = ((_S, _S), (0.0, 1.0), (-_S, _S), (-1.0, 0.0), (-_S, -_S), (0.0, -1.0), (_S, -_S), (1.0, 0.0))
_VEL = [(0.0, 0.0)] + [(v * a, v * b) for v in _SPEED for a, b in _DIR]


def _weights(T):
    """F_0..F_4 of Eqs. 11-13."""
    v2 = [v * v for v in _SPEED]
    out = []
    for k in range(4):
        a, b, c = v2[(k + 1) % 4], v2[(k + 2) % 4], v2[(k + 3) % 4]
        den = v2[k] * (v2[k] - a) * (v2[k] - b) * (v2[k] - c)
        out.append((48.0 * T ** 4 - 6.0 * (a + b + c) * T ** 3 + (a * b + b * c + c * a) * T ** 2
                    - a * b * c / 4.0 * T) / den)
    return [1.0 - 8.0 * (out[0] + out[1] + out[2] + out[3])] + out


def _feq(q, n, ux, uy, T, w):
    vx, vy = _VEL[q]
    b = (ux * ux + uy * uy) / (2.0 * T)
    s = (vx * ux + vy * uy) / T
    br = (1.0 - b) * (1.0 + s + 0.5 * s * s) + 0.5 * b * b + s ** 3 / 6.0 + s ** 4 / 24.0
    return n * w[0 if q == 0 else 1 + (q - 1) // 8] * br


def _mirror(q, axis):
    if q == 0:
        return 0
    k, i = (q - 1) // 8, 1 + (q - 1) % 8
    j = ((8 - i) if axis else (4 - i)) % 8
    return 1 + 8 * k + ((j or 8) - 1)


def _ghosts(f, par, seg, t):
    """Ghost ring of width 2 of f [33, ny + 4, nx + 4] at time t."""
    nx, ny, bc, bs = par["nx"], par["ny"], par["bc"], par["bstate"]

    def state(st):
        st = [torch.tensor(float(a), dtype=torch.float64, device=DEVICE) for a in st]
        w = _weights(st[3])
        return torch.stack([_feq(q, *st, w) for q in range(33)])

    for side in range(4):
        axis, n = (0, nx) if side < 2 else (1, ny)
        for layer in range(2):
            at = (-1 - layer if side % 2 == 0 else n + layer)
            src = {W.PERIODIC: at % n, W.OUTFLOW: 0 if side % 2 == 0 else n - 1,
                   W.WALL: -1 - at if side % 2 == 0 else 2 * n - 1 - at}.get(bc[side], 0)

            def line(pos):
                return f[:, 2:ny + 2, 2 + pos] if axis == 0 else f[:, 2 + pos, 2:nx + 2]

            if bc[side] == W.DIRICHLET:
                line(at).copy_(state(bs[side])[:, None].expand(33, line(at).shape[1]))
            elif bc[side] == W.WALL:
                line(at).copy_(line(src)[[_mirror(q, axis) for q in range(33)]])
            else:
                line(at).copy_(line(src).clone())
            for sside, c0, speed, lower, st in seg:
                if sside == side:
                    c = (np.arange(ny if axis == 0 else nx) + 0.5) * par["dx"]
                    inside = c < c0 + speed * t if lower else ~(c < c0 + speed * t)
                    m = torch.from_numpy(inside).to(DEVICE)
                    line(at)[:, m] = state(st)[:, None]


def _macros(f):
    n, jx, jy, e = (torch.zeros_like(f[0]) for _ in range(4))
    for q, (vx, vy) in enumerate(_VEL):
        n += f[q]
        jx += vx * f[q]
        jy += vy * f[q]
    ux, uy = jx / n, jy / n
    for q, (vx, vy) in enumerate(_VEL):
        e += 0.5 * ((vx - ux) ** 2 + (vy - uy) ** 2) * f[q]
    return n, ux, uy, e / n


def _solve(par, seg, macros, steps):
    nx, ny, flags, lam = par["nx"], par["ny"], par["flags"], par["lam"]
    f = torch.ones((33, ny + 4, nx + 4), dtype=torch.float64, device=DEVICE)
    w = _weights(macros[3])
    for q in range(33):
        f[q, 2:-2, 2:-2] = _feq(q, *macros, w)
    kap, r = par["dt"] / par["dx"], par["dt"] / par["tau"]
    _ghosts(f, par, seg, 0.0)
    for step in range(steps):
        n, ux, uy, T = _macros(f[:, 1:-1, 1:-1])
        P = n * T
        n, ux, uy, T = (a[1:-1, 1:-1] for a in (n, ux, uy, T))
        w = _weights(T)
        nu = []
        for axis, u in ((0, ux), (1, uy)):
            p0 = P[1:-1, 1:-1]
            pp, pm = (P[1:-1, 2:], P[1:-1, :-2]) if axis == 0 else (P[2:, 1:-1], P[:-2, 1:-1])
            ak = (u * kap).abs()
            nu.append(0.5 * lam * ((pp - 2.0 * p0 + pm) / (pp + 2.0 * p0 + pm)).abs() * ak * (1.0 - ak))
        new = torch.empty_like(f)
        for q in range(33):
            p = f[q]
            c0 = p[2:-2, 2:-2]
            acc = c0 + r * (_feq(q, n, ux, uy, T, w) - c0)
            for axis in range(2):
                c = _VEL[q][axis] * kap
                if axis == 0:
                    p1, m1, p2, m2 = p[2:-2, 3:-1], p[2:-2, 1:-3], p[2:-2, 4:], p[2:-2, :-4]
                else:
                    p1, m1, p2, m2 = p[3:-1, 2:-2], p[1:-3, 2:-2], p[4:, 2:-2], p[:-4, 2:-2]
                curv = p1 - 2.0 * c0 + m1
                acc = acc - 0.5 * c * (p1 - m1)
                if not flags & W._NO_LW:
                    acc = acc + 0.5 * c * c * curv
                if not flags & W._NO_DISP:
                    acc = acc + c * (1.0 - c * c) / 12.0 * (p2 - 2.0 * p1 + 2.0 * m1 - m2)
                if not flags & W._NO_VISC:
                    acc = acc + nu[axis] * curv
            new[q, 2:-2, 2:-2] = acc
        f = new
        _ghosts(f, par, seg, (step + 1) * par["dt"])
    f = f[:, 2:-2, 2:-2]
    return _macros(f), f


def _amplification(rows):
    """G of Eq. 18 with the Jacobian of Eq. 20 for rows (n, u1, u2, T, xi_x, xi_y, lambda, flags): [n, 33, 33, 2]."""
    dx, dy, dt, tau = W.VN_SEC4_GRID
    r = dt / tau
    col = [torch.from_numpy(np.array(rows[:, i])).to(DEVICE) for i in range(8)]
    st = [c.clone().requires_grad_(True) for c in col[:4]]  # n, ux, uy, T
    n, ux, uy, T = col[:4]
    G = torch.zeros((len(rows), 33, 33, 2), dtype=torch.float64, device=DEVICE)
    du = torch.stack([torch.stack([torch.ones_like(n), (vx - ux) / n, (vy - uy) / n,
                                   (0.5 * ((vx - ux) ** 2 + (vy - uy) ** 2) - T) / n], 1) for vx, vy in _VEL], 1)
    lw, disp, visc = (1.0 - ((col[7].long() & b) != 0).double() for b in (W._NO_LW, W._NO_DISP, W._NO_VISC))
    for q in range(33):
        g = torch.autograd.grad(_feq(q, *st, _weights(st[3])).sum(), st)
        G[:, q, :, 0] = r * sum(g[a][:, None] * du[:, :, a] for a in range(4))
        G[:, q, q, 0] += 1.0 - r
        for v, u, h, xi in ((_VEL[q][0], ux, dx, col[4]), (_VEL[q][1], uy, dy, col[5])):
            c, k = v * dt / h, (u * dt / h).abs()
            curv = torch.cos(xi) - 1.0
            G[:, q, q, 0] += lw * c * c * curv + visc * col[6] * k * (1.0 - k) * curv
            G[:, q, q, 1] += -c * torch.sin(xi) + disp * c * (1.0 - c * c) / 6.0 * (torch.sin(2.0 * xi) - 2.0 * torch.sin(xi))
    return G


def exact(case, seed):
    if case["kind"] == "vn":  # 64-bit arithmetic does not determine the spectra, only the matrices
        return {"max_abs": None, "G": _amplification(_vn_rows(case, seed)), "status": None}
    if case["kind"] == "batch":
        got = []
        for sub, s in _batch_members(case, seed):
            par, seg, f = _problem(sub, s)
            got.append(torch.stack(_solve(par, seg, f, case["steps"])[0]).reshape(4, -1))
        return {"macros": torch.cat(got, 1)}
    par, seg, f = _problem(case, seed)
    m, f = _solve(par, seg, f, case["steps"])
    out = {"rho": m[0], "u": m[1], "v": m[2], "T": m[3]}
    if case.get("prec") != "fneq32":
        out["f"] = f
    return out
