"""Performance cases of the library: what its users have it do.

Each case is one call (or one short sequence of calls) of the public API on
inputs of the repository's own configurations, or of sizes around them:

  riemann_1d_f64   the 1D two-state Riemann problem in FP64, 400 cells, the
                   device time loop: the smallest call, launches and latency
  shear_2d_f32     the 2D shear layer, device time loop
  smooth_3d_f32    the periodic smooth flow at 256^3 in FP32: the bulk path
  smooth_3d_f64    the same flow in FP64: the parity path
  blast_3d_f32     the strong blast at 512^3 between reflecting walls, with
                   the conserved totals logged each step: the largest run
  ragged_3d_f32    a 3D mesh whose rows are no multiple of 16 bytes
  weno_3d_f32      the paper's own scheme, WENO5-Z + HLL
  batch_f32        4096 independent 1D / 2D problems in one launch
  gradient_2d_f32  gradients of a density misfit through a rollout
  advection_f32, diffusion_f32, exchange_f32
                   the three radiation operators of the split

`draw` gives further cases of the same kinds: other extents (odd ones among
them), boundary kinds, element types and flows.  `exact` restates the scheme
in plain 64-bit torch.
"""
import math
import random

import numpy as np
import torch

import paper_2509_08971_gb300 as hh
from paper_2509_08971_gb300.autograd import Mesh, rollout

BC = {"periodic": 0, "outflow": 1, "reflect": 2}
DTYPE = {"f32": torch.float32, "f64": torch.float64}
# c = kappa = 1 of the diffusion; CGS constants of the heating / cooling test
C_LIGHT, KAPPA, A_RAD, CV = 2.99792458e10, 0.4, 7.565733250033928e-15, 2.078615655e8
MODES = ((0, 0, 1), (0, 1, 0), (1, 0, 0), (0, 1, 1), (0, 1, -1), (1, 0, 1), (1, 0, -1), (1, 1, 0))


def _advance(name, shape, dtype, flow, bc, steps, scheme="plm", totals=False):
    nz, ny, nx = shape
    return {"name": name, "kind": "advance", "nx": nx, "ny": ny, "nz": nz, "dtype": dtype,
            "flow": flow, "bc": bc, "steps": steps, "scheme": scheme, "totals": totals}


def _operator(name, kind, shape, dtype, bc, **more):
    nz, ny, nx = shape
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "bc": bc, **more}


def listed():
    cube = (256, 256, 256)
    return [
        # the 1D convergence study's problem: 400 cells to t = 0.15
        _advance("riemann_1d_f64", (1, 1, 400), "f64", "riemann", "outflow", 100),
        # forward runs of the shear layer that the gradients are taken of
        _advance("shear_2d_f32", (1, 256, 256), "f32", "shear", "periodic", 50),
        # the smooth-flow convergence and conservation runs, bulk and parity precision
        _advance("smooth_3d_f32", cube, "f32", "smooth", "periodic", 4),
        _advance("smooth_3d_f64", (128, 128, 128), "f64", "smooth", "periodic", 2),
        # the production run: a strong blast in a box, conservation watched
        _advance("blast_3d_f32", (512, 512, 512), "f32", "blast", "reflect", 2, totals=True),
        # a mesh that nobody rounded to the hardware
        _advance("ragged_3d_f32", (93, 117, 150), "f32", "smooth", "outflow", 8),
        # the paper's scheme
        _advance("weno_3d_f32", cube, "f32", "smooth", "periodic", 2, scheme="weno"),
        # parameter studies: thousands of small problems
        {"name": "batch_f32", "kind": "batch", "problems": 4096, "min1d": 64, "max1d": 4096,
         "min2d": 32, "max2d": 256, "mix": 0, "dtype": "f32", "steps": 5},
        # fitting an initial state and gamma
        {"name": "gradient_2d_f32", "kind": "gradient", "nx": 256, "ny": 256, "dtype": "f32",
         "bc": "periodic", "steps": 20, "every": 10},
        # the radiation operators, called once per hydro step
        _operator("advection_f32", "advection", cube, "f32", "periodic"),
        _operator("diffusion_f32", "diffusion", cube, "f32", "periodic", number=300.0, rtol=1e-5,
                  cycles=40),
        _operator("exchange_f32", "exchange", cube, "f32", "periodic"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["1d", "2d", "3d", "3d", "3d", "weno", "batch", "gradient", "advection",
                       "diffusion", "exchange"])
    bc = rng.choice(["periodic", "outflow", "reflect"])
    dtype = rng.choice(["f32", "f32", "f64"])
    small = dtype == "f64"
    if kind == "1d":
        c = _advance("", (1, 1, _log(rng, 64, 4096)), dtype, "riemann", "outflow", 100)
    elif kind == "2d":
        hi = 256 if small else 1024
        c = _advance("", (1, _log(rng, 32, hi), _log(rng, 32, hi)), dtype, "shear", bc, 20)
    elif kind in ("3d", "weno"):
        hi = 80 if small else (200 if kind == "weno" else 320)
        c = _advance("", tuple(_log(rng, 16, hi) for _ in range(3)), dtype,
                     "smooth" if kind == "weno" else rng.choice(["smooth", "blast"]), bc, 1 if small else 2,
                     scheme="weno" if kind == "weno" else "plm", totals=rng.random() < 0.5)
    elif kind == "batch":
        c = {"kind": kind, "problems": _log(rng, 16, 64 if small else 1024),
             "min1d": rng.choice([16, 64]), "max1d": _log(rng, 256, 4096),
             "min2d": rng.choice([8, 32]), "max2d": _log(rng, 64, 128 if small else 256),
             "mix": rng.randrange(1000), "dtype": dtype, "steps": rng.choice([2, 5])}
    elif kind == "gradient":
        hi = 128 if small else 384
        c = {"kind": kind, "nx": _log(rng, 32, hi), "ny": _log(rng, 32, hi), "dtype": dtype,
             "bc": bc, "steps": 10, "every": rng.choice([4, 10])}
    else:
        hi = {"advection": 320, "diffusion": 160, "exchange": 320}[kind]
        n = tuple(_log(rng, 16, 96 if small else hi) for _ in range(3))
        c = _operator("", kind, n, dtype, bc)
        if kind == "diffusion":
            c.update(number=float(_log(rng, 1, 300)), rtol=1e-7 if small else 1e-4, cycles=10)
    c.pop("name", None)
    return c


# ------------------------------------------------------------------- inputs --

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _rand(shape, g, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") * (hi - lo) + lo


def _cons(rho, u, v, w, p, gamma):
    E = p / (gamma - 1.0) + 0.5 * rho * (u * u + v * v + w * w)
    return torch.stack(torch.broadcast_tensors(rho, rho * u, rho * v, rho * w, E))


def _centres(n, shape):
    return ((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n).view(shape)


def _gamma(case):
    return 5.0 / 3.0 if case.get("flow") == "smooth" or case["kind"] not in ("advance", "gradient", "batch") else 1.4


def _cfl(case):
    return 0.3 if case.get("flow") == "blast" else 0.4


def _state(case, seed):
    """Initial conserved state (5, nz, ny, nx), FP64, on the unit box."""
    nz, ny, nx = case.get("nz", 1), case["ny"] if "ny" in case else 1, case["nx"]
    x, y, z = _centres(nx, (1, 1, nx)), _centres(ny, (1, ny, 1)), _centres(nz, (nz, 1, 1))
    full, gamma, flow, g, r = (nz, ny, nx), _gamma(case), case.get("flow", "smooth"), _gen(seed), random.Random(seed)
    zero, one = torch.zeros(full, dtype=torch.float64, device="cuda"), torch.ones(full, dtype=torch.float64, device="cuda")
    if flow == "riemann":
        while True:
            rl, rr, pl, pr = (math.exp(r.uniform(math.log(0.1), math.log(10.0))) for _ in range(4))
            ul, ur = r.uniform(-1, 1), r.uniform(-1, 1)
            if 2.0 * (math.sqrt(gamma * pl / rl) + math.sqrt(gamma * pr / rr)) / (gamma - 1.0) > ur - ul:
                break
        left = x + zero <= 0.5
        pick = lambda a, b: torch.where(left, a * one, b * one)  # noqa: E731
        return _cons(pick(rl, rr), pick(ul, ur), zero, zero, pick(pl, pr), gamma)
    if flow == "shear":
        inside = (y - 0.5).abs() + zero < 0.25
        # the configuration's layer, with sound waves and the cell noise of a state that has run
        rho = torch.where(inside, 2.0 * one, one) + 1e-3 * _rand(full, g, -1, 1)
        v = 0.01 * sum(r.uniform(-1, 1) * torch.sin(2 * math.pi * m * x + r.uniform(0, 2 * math.pi)) for m in range(1, 5))
        wave = 0.2 * torch.sin(2 * math.pi * (x + y) + r.uniform(0, 7)) + 0.1 * torch.sin(2 * math.pi * (2 * x - y) + r.uniform(0, 7))
        noise = lambda: 1e-3 * _rand(full, g, -1, 1)  # noqa: E731
        return _cons(rho, torch.where(inside, 0.5 * one, -0.5 * one) + noise(), v + noise(), zero, 2.5 + wave + noise(), gamma)
    if flow == "blast":
        rho, p = 1.0 + 0.01 * _rand(full, g, -1, 1), 1e-5 * one
        U = _cons(rho, zero, zero, zero, p, gamma)
        h = [max(4.0 / n, 0.0) for n in (nx, ny, nz)]
        hot = ((x - 0.5) / h[0]) ** 2 + ((y - 0.5) / h[1]) ** 2 + ((z - 0.5) / h[2]) ** 2 <= 1.0 + 1e-12
        U[4] += torch.where(hot, 1.0 / (hot.sum().double() / (nx * ny * nz)), 0.0)
        return U
    rho = 1.0 + 0.2 * torch.sin(2 * math.pi * (x + y + z))
    u, v, w, p = one.clone(), one.clone(), one.clone(), one.clone()
    cs = math.sqrt(gamma)
    for kx, ky, kz in MODES:
        norm = math.sqrt(kx * kx + ky * ky + kz * kz)
        d = 1e-3 * torch.sin(2 * math.pi * (kx * x + ky * y + kz * z) + r.uniform(0, 2 * math.pi))
        rho, p = rho + d, p + cs * cs * d
        u, v, w = u + kx / norm * cs * d, v + ky / norm * cs * d, w + kz / norm * cs * d
    return _cons(rho, u, v, w, p, gamma)


def _batch(case, seed):
    """Extents of the problems (the case's) and, per problem, four (rho, u, v, p) states."""
    r = np.random.default_rng(case["mix"])
    n, n1 = case["problems"], case["problems"] // 2
    nx, ny = np.empty(n, dtype=np.int64), np.ones(n, dtype=np.int64)
    nx[:n1] = r.integers(case["min1d"], case["max1d"] + 1, n1)
    nx[n1:] = ny[n1:] = r.integers(case["min2d"], case["max2d"] + 1, n - n1)
    r = np.random.default_rng(seed)
    rho, p = (np.exp(r.uniform(math.log(0.1), math.log(10.0), (n, 4))) for _ in range(2))
    u, v = r.uniform(-1, 1, (n, 4)), r.uniform(-1, 1, (n, 4)) * (ny > 1)[:, None]
    return nx, ny, np.stack([rho, u, v, p])


def _batch_cells(nx, ny):
    """Problem, x and y of every cell of the batch, problem after problem."""
    nx, ny = torch.as_tensor(nx, device="cuda"), torch.as_tensor(ny, device="cuda")
    prob = torch.repeat_interleave(torch.arange(len(nx), device="cuda"), nx * ny)
    first = torch.cumsum(nx * ny, 0) - nx * ny
    c = torch.arange(len(prob), device="cuda") - first[prob]
    return prob, c % nx[prob], c // nx[prob], nx, ny, first


def _batch_state(prob, x, y, nx, ny, states, gamma):
    quad = ((x + 0.5) / nx[prob] > 0.5).long() + 2 * ((y + 0.5) / ny[prob] > 0.5).long() * (ny[prob] > 1).long()
    rho, u, v, p = (torch.as_tensor(s, device="cuda")[prob, quad] for s in states)
    return _cons(rho, u, v, torch.zeros_like(rho), p, gamma)


def _offsets(nx, ny):
    """Element offset of each problem in the packed state (rounded up to 32) and its length."""
    n = 5 * nx * ny
    up = (n + 31) // 32 * 32
    return np.cumsum(up) - up, int(up.sum())


def _packed_index(prob, x, y, nx, ny, off):
    off = torch.as_tensor(off, device="cuda")
    at = off[prob] + y * nx[prob] + x
    return at, (nx * ny)[prob]


def _target(case, seed):
    r = random.Random(seed + 7919)
    x, y = _centres(case["nx"], (1, 1, -1)), _centres(case["ny"], (1, -1, 1))
    f = torch.zeros((1, case["ny"], case["nx"]), dtype=torch.float64, device="cuda")
    for m in range(1, 5):
        a, b, px, py = r.uniform(-1, 1), r.uniform(-1, 1), r.uniform(0, 7), r.uniform(0, 7)
        f = f + 0.25 * (a * torch.sin(2 * math.pi * m * x + px) + b * torch.sin(2 * math.pi * m * y + py))
    return 1.5 + 0.1 * f


def _inputs(case, seed):
    """The case's tensors in the case's element type."""
    dt = DTYPE[case["dtype"]]
    kind = case["kind"]
    if kind == "advance":
        return {"U": _state(case, seed).to(dt)}
    if kind == "gradient":
        U = _state(dict(case, flow="shear", nz=1), seed).to(dt)
        step = 0.4 / _rate(U.double(), _mesh(dict(case, nz=1)), 1.4).item()
        return {"U": U, "target": _target(case, seed).to(dt), "dts": [step] * case["steps"]}
    shape, g = (case["nz"], case["ny"], case["nx"]), _gen(seed)
    if kind == "exchange":
        # Sec. 3.2 cooling: rho, T_f, T_r spread by +-50 %, a moving fluid
        f = lambda: torch.exp(_rand(shape, g, -1, 1) * math.log1p(0.5))  # noqa: E731
        rho, Tf, Tr = 1e-7 * f(), 1.1e9 * f(), 3.4e6 * f()
        v = _rand((3,) + shape, g, -1e5, 1e5)
        e = rho * CV * Tf + 0.5 * rho * (v * v).sum(0)
        return {"U": torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], e]).to(dt), "E": (A_RAD * Tr ** 4).to(dt)}
    U = _state(case, seed)
    if kind == "diffusion":
        U[0] = _rand(shape, g, 1.0, 1.5)
    return {"U": U.to(dt), "E": _rand(shape, g, 1.0, 1.5).to(dt)}


def _mesh(case):
    n = (case["nx"], case["ny"], case.get("nz", 1))
    return {"n": n, "dx": [1.0 / k for k in n], "bc": BC[case["bc"]]}


def _diffusion_dt(case):
    return case["number"] / max(case["nx"], case["ny"], case["nz"]) ** 2


def _advection_dt(case, U):
    return 0.4 / _rate(U.double(), _mesh(case), _gamma(case)).item()


def prepare(case, seed):
    kind, dt = case["kind"], DTYPE[case["dtype"]]
    if kind == "batch":
        nx, ny, states = _batch(case, seed)
        prob, x, y, tx, ty, _ = _batch_cells(nx, ny)
        U = _batch_state(prob, x, y, tx, ty, states, 1.4).to(dt)
        B = hh.HardBatch(nx, ny, 1.4, hh.HARD_BC_OUTFLOW, dtype=dt)
        first = B.empty()
        at, stride = _packed_index(prob, x, y, tx, ty, B.offsets)
        for f in range(5):
            first[at + f * stride] = U[f]
        return {"case": case, "B": B, "U0": first, "U": first.clone(), "t": torch.zeros(len(nx), dtype=torch.float64, device="cuda")}
    got = _inputs(case, seed)
    if kind == "gradient":
        gamma = torch.tensor(1.4, dtype=dt, device="cuda", requires_grad=True)
        mesh = Mesh((1, case["ny"], case["nx"]), BC[case["bc"]])
        return {"case": case, "U0": got["U"].requires_grad_(), "gamma": gamma, "mesh": mesh, "target": got["target"], "dts": got["dts"]}
    m = hh.HardHydro((case["nz"], case["ny"], case["nx"]), _gamma(case), BC[case["bc"]], dtype=dt,
                     scheme=hh.HARD_SCHEME_WENO5Z_HLL if case.get("scheme") == "weno" else hh.HARD_SCHEME_PLM_HLLC)
    s = {"case": case, "m": m, "U": got["U"]}
    if kind == "advance":
        s["U0"], s["U"] = got["U"], got["U"].clone()
    else:
        s["E0"], s["E"] = got["E"], got["E"].clone()
    if kind == "advection":
        s["dt"] = _advection_dt(case, got["U"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "advance":
        # a run from its initial state; the time as the state's type
        s["U"].copy_(s["U0"])
        t, _, _ = s["m"].advance(s["U"], case["steps"], _cfl(case), t_end=0.15 if case["flow"] == "riemann" else 0.0,
                                 log_totals=case["totals"])
        return {"U": s["U"], "t": t.to(s["U"].dtype)}
    if kind == "batch":
        s["U"].copy_(s["U0"])
        s["t"].zero_()
        t = s["B"].step(s["U"], case["steps"], 0.4, t=s["t"])
        return {"U": s["U"], "t": t.to(s["U"].dtype)}
    if kind == "gradient":
        U0, gamma = s["U0"], s["gamma"]
        U0.grad = gamma.grad = None
        U = rollout(U0, gamma, s["mesh"], s["dts"], case["every"])
        (U[0] - s["target"]).square().mean().backward()
        return {"U": U.detach(), "dU": U0.grad, "dgamma": gamma.grad}
    if kind == "exchange":
        # in place, as between two hydro steps: each call is a fresh implicit step
        s["m"].rad_exchange(s["U"], s["E"], 1e-12, C_LIGHT, KAPPA, A_RAD, CV)
        return {"E_total": s["U"][4], "E": s["E"]}
    s["E"].copy_(s["E0"])
    if kind == "advection":
        s["m"].advect_E(s["U"], s["E"], s["dt"])
    else:
        s["m"].fld_step(s["U"], s["E"], _diffusion_dt(case), 1.0, 1.0, rtol=case["rtol"], max_cycles=case["cycles"])
    return {"E": s["E"]}


def work(case):
    """Bytes: the state read and written once per step (a rollout's gradient: its steps
    forward and backward).  Operations: the scheme's arithmetic per cell and stage."""
    size = 4 if case["dtype"] == "f32" else 8
    kind = case["kind"]
    if kind == "batch":
        m1, m2 = (case["min1d"] + case["max1d"]) / 2, (case["min2d"] ** 2 + case["min2d"] * case["max2d"] + case["max2d"] ** 2) / 3
        cells, steps = case["problems"] / 2 * (m1 + m2), case["steps"]
        return {"bytes": 10.0 * size * cells * steps, "flops": 2.0 * steps * cells * 250}
    cells = case["nx"] * case["ny"] * case.get("nz", 1)
    axes = sum(case.get(k, 1) > 1 for k in ("nx", "ny", "nz"))
    if kind == "advance":
        face = 360 if case["scheme"] == "weno" else 120
        return {"bytes": 10.0 * size * cells * case["steps"], "flops": 2.0 * case["steps"] * cells * (30 + axes * face)}
    if kind == "gradient":
        return {"bytes": 30.0 * size * cells * case["steps"], "flops": 2.0 * case["steps"] * cells * (60 + axes * 500)}
    if kind == "exchange":
        return {"bytes": 8.0 * size * cells, "flops": 100.0 * cells}
    if kind == "advection":
        return {"bytes": 6.0 * size * cells, "flops": 2.0 * cells * axes * 135}
    return {"bytes": 3.0 * size * cells, "flops": 4.0 * cells * 8 / 7 * 4 * 26}


# -------------------------------------------- the same results, 64-bit torch --

def _ghosts(lo, hi, n, bc):
    """Source index and sign of the normal momentum of cells lo..hi-1 of an axis."""
    idx, sign = [], []
    for m in range(lo, hi):
        inside = 0 <= m < n
        idx.append(m if inside else m % n if bc == 0 else min(max(m, 0), n - 1) if bc == 1 else (-1 - m if m < 0 else 2 * n - 1 - m))
        sign.append(-1.0 if bc == 2 and not inside else 1.0)
    return torch.tensor(idx, device="cuda"), torch.tensor(sign, dtype=torch.float64, device="cuda")


def _prim(U, gamma):
    u, v, w = U[1] / U[0], U[2] / U[0], U[3] / U[0]
    return torch.stack([U[0], u, v, w, (gamma - 1.0) * (U[4] - 0.5 * U[0] * (u * u + v * v + w * w))])


def _rate(U, mesh, gamma):
    W = _prim(U, gamma)
    c = torch.sqrt(gamma * W[4] / W[0])
    return sum((W[1 + d].abs() + c) / mesh["dx"][d] for d in range(3) if mesh["n"][d] > 1).max()


def _minmod(a, b):
    return torch.where(a * b > 0, torch.where(a.abs() <= b.abs(), a, b), torch.zeros_like(a))


def _flux(W, d, gamma):
    """Conserved state and physical flux along axis d of primitives W."""
    rho, v, p = W[0], W[1:4], W[4]
    E = p / (gamma - 1.0) + 0.5 * rho * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])
    U = torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], E])
    P = [torch.zeros_like(p)] * 5
    P[1 + d], P[4] = p, p * v[d]
    return U, U * v[d] + torch.stack(P)


def _speeds(L, R, d, gamma):
    cL, cR = torch.sqrt(gamma * L[4] / L[0]), torch.sqrt(gamma * R[4] / R[0])
    return torch.minimum(L[1 + d] - cL, R[1 + d] - cR), torch.maximum(L[1 + d] + cL, R[1 + d] + cR)


def _hllc(L, R, d, gamma):
    SL, SR = _speeds(L, R, d, gamma)
    mL, mR = L[0] * (SL - L[1 + d]), R[0] * (SR - R[1 + d])
    S = (R[4] - L[4] + mL * L[1 + d] - mR * R[1 + d]) / (mL - mR)
    left = S >= 0
    W, m, SK = torch.where(left, L, R), torch.where(left, mL, mR), torch.where(left, SL, SR)
    U, F = _flux(W, d, gamma)
    star = torch.where(left, SL < 0, SR > 0)
    one = torch.ones_like(m)
    m = torch.where(star, m, one)
    fac = m / torch.where(star, SK - S, one)
    parts = [fac, fac * W[1], fac * W[2], fac * W[3], fac * (U[4] / W[0] + (S - W[1 + d]) * (S + W[4] / m))]
    parts[1 + d] = fac * S
    return torch.where(star, F + SK * (torch.stack(parts) - U), F)


def _weno(a, b, c, d, e):
    p = ((2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6)
    q = ((a - 2 * b + c, a - 4 * b + 3 * c), (b - 2 * c + d, b - d), (c - 2 * d + e, 3 * c - 4 * d + e))
    beta = [13.0 / 12.0 * s * s + 0.25 * t * t for s, t in q]
    tau = (beta[0] - beta[2]).abs()
    w = [k * (1 + tau / (x + 1e-30)) for k, x in zip((0.1, 0.6, 0.3), beta)]
    return (w[0] * p[0] + w[1] * p[1] + w[2] * p[2]) / (w[0] + w[1] + w[2])


def _hll(L, R, d, gamma):
    SL, SR = _speeds(L, R, d, gamma)
    SL, SR = SL.clamp(max=0.0), SR.clamp(min=0.0)
    (UL, FL), (UR, FR) = _flux(L, d, gamma), _flux(R, d, gamma)
    return (SR * FL - SL * FR + SL * SR * (UR - UL)) / (SR - SL)


def _faces(W, dim, n, scheme):
    """Left and right states of the n + 1 faces of an axis from its padded cells."""
    at = lambda k, m=n + 1: W.narrow(dim, k, m)  # noqa: E731
    if scheme == "weno":
        return _weno(at(0), at(1), at(2), at(3), at(4)), _weno(at(5), at(4), at(3), at(2), at(1))
    d = at(1, n + 3) - at(0, n + 3)
    s = 0.5 * _minmod(d.narrow(dim, 0, n + 2), d.narrow(dim, 1, n + 2))
    return at(1) + s.narrow(dim, 0, n + 1), at(2) - s.narrow(dim, 1, n + 1)


def _padded(U, d, k0, k1, g, mesh, momentum=True):
    """Planes k0..k1-1 of U with g ghost cells on both sides along axis d."""
    n, dim = mesh["n"][d], U.dim() - 1 - d
    idx, sign = _ghosts(k0 - g, k1 + g, n, mesh["bc"]) if d == 2 else _ghosts(-g, n + g, n, mesh["bc"])
    P = (U if d == 2 else U.narrow(-3, k0, k1 - k0)).index_select(dim, idx)
    if momentum and mesh["bc"] == 2:
        shape = [5, 1, 1, 1]
        shape[dim] = len(idx)
        flip = torch.ones(shape, dtype=torch.float64, device="cuda")
        flip[1 + d] = sign.view(shape[1:])
        P = P * flip
    return P


def _chunks(n):
    return max(1, (1 << 22) // (n[0] * n[1]))


def _rhs(U, mesh, gamma, scheme):
    n, g = mesh["n"], 3 if scheme == "weno" else 2
    out, dz = [], _chunks(mesh["n"])
    for k0 in range(0, n[2], dz):
        k1, L = min(k0 + dz, n[2]), 0.0
        for d in range(3):
            if n[d] < 2:
                continue
            dim, m = 3 - d, k1 - k0 if d == 2 else n[d]
            qL, qR = _faces(_prim(_padded(U, d, k0, k1, g, mesh), gamma), dim, m, scheme)
            F = _hll(qL, qR, d, gamma) if scheme == "weno" else _hllc(qL, qR, d, gamma)
            L = L - (F.narrow(dim, 1, m) - F.narrow(dim, 0, m)) / mesh["dx"][d]
        out.append(L)
    return torch.cat(out, 1) if len(out) > 1 else out[0]


def _step(U, dt, mesh, gamma, scheme):
    U1 = U + dt * _rhs(U, mesh, gamma, scheme)
    return 0.5 * U + 0.5 * (U1 + dt * _rhs(U1, mesh, gamma, scheme))


def _exact_advance(case, seed):
    U, mesh, t = _inputs(case, seed)["U"].double(), _mesh(case), 0.0
    end = 0.15 if case["flow"] == "riemann" else 0.0
    for _ in range(case["steps"]):
        dt = _cfl(case) / _rate(U, mesh, _gamma(case)).item()
        if end:
            dt = max(0.0, min(dt, end - t))
        if dt > 0:
            U = _step(U, dt, mesh, _gamma(case), case["scheme"])
        t += dt
    return {"U": U, "t": torch.tensor(t, dtype=torch.float64)}


def _exact_gradient(case, seed):
    got, mesh = _inputs(case, seed), _mesh(dict(case, nz=1))
    gamma = torch.tensor(1.4, dtype=DTYPE[case["dtype"]], device="cuda").double()
    states, target = [got["U"].double()], got["target"].double()
    for dt in got["dts"]:
        states.append(_step(states[-1], dt, mesh, gamma, "plm"))
    g = torch.zeros_like(states[-1])
    g[0] = 2.0 * (states[-1][0] - target) / target.numel()
    dgamma = torch.zeros_like(gamma)
    for U, dt in zip(reversed(states[:-1]), reversed(got["dts"])):
        U, gm = U.clone().requires_grad_(), gamma.clone().requires_grad_()
        g, dg = torch.autograd.grad(_step(U, dt, mesh, gm, "plm"), (U, gm), g)
        dgamma = dgamma + dg
    return {"U": states[-1], "dU": g, "dgamma": dgamma}


def _exact_batch(case, seed):
    nx, ny, states = _batch(case, seed)
    prob, x, y, tx, ty, first = _batch_cells(nx, ny)
    U = _batch_state(prob, x, y, tx, ty, states, 1.4).to(DTYPE[case["dtype"]]).double()
    dx, two, P = (1.0 / tx.double(), 1.0 / ty.double()), ty > 1, len(nx)

    def rhs(U):
        L = torch.zeros_like(U)
        W = _prim(U, 1.4)
        for a in range(0, U.shape[1], 1 << 23):
            s = slice(a, min(a + (1 << 23), U.shape[1]))
            p, cx, cy = prob[s], x[s], y[s]
            for d in range(2):
                def cell(k):  # the cells k along axis d, the edge cell repeated
                    X = (cx + k).clamp(min=0).minimum(tx[p] - 1) if d == 0 else cx
                    Y = (cy + k).clamp(min=0).minimum(ty[p] - 1) if d == 1 else cy
                    return W[:, first[p] + Y * tx[p] + X]
                q = [cell(k) for k in range(-2, 3)]
                e = [q[k + 1] - q[k] for k in range(4)]
                sl = [0.5 * _minmod(e[k], e[k + 1]) for k in range(3)]
                F = [_hllc(q[1 + k] + sl[k], q[2 + k] - sl[k + 1], d, 1.4) for k in range(2)]
                L[:, s] -= torch.where(two[p] if d else torch.ones_like(two[p]), (F[1] - F[0]) / dx[d][p], 0.0)
        return L

    t = torch.zeros(P, dtype=torch.float64, device="cuda")
    for _ in range(case["steps"]):
        W = _prim(U, 1.4)
        c = torch.sqrt(1.4 * W[4] / W[0])
        r = (W[1].abs() + c) / dx[0][prob] + torch.where(two[prob], (W[2].abs() + c) / dx[1][prob], 0.0)
        dt = 0.4 / torch.zeros_like(t).scatter_reduce(0, prob, r, "amax")
        del W, c, r
        U1 = U + dt[prob] * rhs(U)
        U = 0.5 * U + 0.5 * (U1 + dt[prob] * rhs(U1))
        t = t + dt
    off, length = _offsets(nx, ny)
    packed = torch.zeros(length, dtype=torch.float64, device="cuda")
    at, stride = _packed_index(prob, x, y, tx, ty, off)
    for f in range(5):
        packed[at + f * stride] = U[f]
    return {"U": packed, "t": t}


def _exact_exchange(case, seed):
    got = _inputs(case, seed)
    U, Er = got["U"].double(), got["E"].double()
    kin = 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / U[0]
    e, k, rcv = U[4] - kin, 1e-12 * C_LIGHT * KAPPA * U[0], U[0] * CV
    total = e + Er
    # x - e = k (total - x - a T^4) increases in x and is convex: Newton from the right
    x = torch.minimum(total, rcv * ((e + k * total) / (k * A_RAD)) ** 0.25)
    for _ in range(60):
        aT4 = A_RAD * (x / rcv) ** 4
        x = x - (x - e - k * (total - x - aT4)) / (1 + k * (1 + 4 * aT4 / x))
    return {"E_total": x + kin, "E": Er + (e - x)}


def _exact_advection(case, seed):
    got, mesh, n = _inputs(case, seed), _mesh(case), (case["nx"], case["ny"], case["nz"])
    dt, E0 = _advection_dt(case, got["U"]), got["E"].double()
    U = got["U"].double()

    def rhs(E):
        out, dz = [], _chunks(n)
        for k0 in range(0, n[2], dz):
            k1, L = min(k0 + dz, n[2]), 0.0
            for d in range(3):
                dim, m = 2 - d, k1 - k0 if d == 2 else n[d]
                P = _padded(U, d, k0, k1, 3, mesh)
                (eL, eR), (uL, uR) = (_faces(q, dim, m, "weno") for q in (_padded(E, d, k0, k1, 3, mesh, False), P[1 + d] / P[0]))
                F = 0.5 * (eL * uL + eR * uR) - 0.5 * torch.maximum(uL.abs(), uR.abs()) * (eR - eL)
                L = L - (F.narrow(dim, 1, m) - F.narrow(dim, 0, m)) / mesh["dx"][d]
            out.append(L)
        return torch.cat(out, 0)

    E1 = E0 + dt * rhs(E0)
    return {"E": 0.5 * E0 + 0.5 * (E1 + dt * rhs(E1))}


def _exact_diffusion(case, seed):
    got, n, per = _inputs(case, seed), (case["nx"], case["ny"], case["nz"]), case["bc"] == "periodic"
    E0, rho, dt = got["E"].double(), got["U"][0].double(), _diffusion_dt(case)

    def shift(q, d, s):  # the neighbour of every cell, the edge cell repeated at a wall
        if per:
            return q.roll(-s, 2 - d)
        return q.index_select(2 - d, (torch.arange(n[d], device="cuda") + s).clamp(0, n[d] - 1))

    grad = sum(((shift(E0, d, 1) - shift(E0, d, -1)) * (0.5 * n[d])) ** 2 for d in range(3))
    R = grad.sqrt() / (rho * E0)
    D = (2 + R) / (6 + 3 * R + R * R) / rho
    w = [0.5 * dt * n[d] ** 2 * (D + shift(D, d, 1)) for d in range(3)]
    if not per:
        for d in range(3):
            w[d].select(2 - d, n[d] - 1).zero_()

    def apply(q):
        out = q.clone()
        for d in range(3):
            flux = w[d] * (shift(q, d, 1) - q)
            low = flux.roll(1, 2 - d)  # the last face of a wall carries nothing
            out -= flux - low
        return out

    x, r = E0.clone(), E0 - apply(E0)
    p, rr = r.clone(), (r * r).sum()
    stop = 1e-26 * (E0 * E0).sum()
    for k in range(4000):
        q = apply(p)
        a = rr / (p * q).sum()
        x, r = x + a * p, r - a * q
        new = (r * r).sum()
        if k % 20 == 0 and new < stop:
            break
        p, rr = r + (new / rr) * p, new
    return {"E": x}


def exact(case, seed):
    with torch.no_grad() if case["kind"] != "gradient" else torch.enable_grad():
        return {"advance": _exact_advance, "batch": _exact_batch, "gradient": _exact_gradient,
                "exchange": _exact_exchange, "advection": _exact_advection,
                "diffusion": _exact_diffusion}[case["kind"]](case, seed)
