"""Performance cases of the hydrodynamics step: what a program that uses this library has it do.

A case is a dict of plain values.  `prepare` makes what such a program holds before the call (a solver with its
state, host buffers, an ensemble, a trained network), `run` is one pass through the public entry points of
`paper_1306_6883_gb300.solver`, `work` says what a pass cannot do without, and `exact` gives the outputs in 64 bits
from plain torch operations.

Keys of a case:
  kind       "advance" (steps kept on the device), "loop" (the paper's driver loop with the time step on the host),
             "host" (state in pinned host memory, each step up and down) or "ensemble"
  problem    "sod", "kh", "sedov", "rt" or "quad"; sizes nx, ny (ensembles: members, and seed-drawn sizes up to nx)
  precision  "fp32" or "fp64"
  steps      time steps of one pass
  split, riemann ("two-shock" | "hllc"), recon ("plm" | "ppm"), learned: the options of the step
  fresh      the pass starts by uploading the initial state (problems that would run out of their domain)
"""
import math

import numpy as np
import torch

from paper_1306_6883_gb300 import hydro as H
from paper_1306_6883_gb300.solver import Ensemble, Model, Solver

NG = 4
GAMMA = 1.4
CFL = 0.8
PERIODIC, OUTFLOW, HYDROSTATIC = "periodic", "outflow", "hydrostatic"
MEMBER_SIZES = (64, 128, 256, 512)
DEVICE = "cuda"


def _case(name, kind, problem, nx, ny, precision, steps, split=0, riemann="two-shock", recon="plm", learned=False,
          fresh=False, members=0):
    c = {"kind": kind, "problem": problem, "nx": nx, "ny": ny, "precision": precision, "steps": steps, "split": split,
         "riemann": riemann, "recon": recon, "learned": learned, "fresh": fresh, "members": members}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the paper's own driver loop on its shock tube at its size, in the default precision: fill ghosts, read
        # the time step on the host, step (the smallest call, bound by latency)
        _case("sod 128 fp64 host loop", "loop", "sod", 128, 128, "fp64", 8, fresh=True),
        # a small exploratory run, one chunk of the command-line driver's steps
        _case("kh 64 fp32", "advance", "kh", 64, 64, "fp32", 32),
        # the shear layer at the size it is compared at, in both precisions
        _case("kh 1024 fp64", "advance", "kh", 1024, 1024, "fp64", 2),
        _case("kh 1024 fp32", "advance", "kh", 1024, 1024, "fp32", 10),
        # the blast of the FP32 accuracy comparison
        _case("sedov 4096 fp32", "advance", "sedov", 4096, 4096, "fp32", 4),
        # the largest run, its Riemann iterations started by the trained network
        _case("sedov 8192 fp32 learned", "advance", "sedov", 8192, 8192, "fp32", 1, learned=True),
        # gravity, hydrostatic walls and a ragged grid
        _case("rt 317x951 fp32", "advance", "rt", 317, 951, "fp32", 20, fresh=True),
        # the other forms of the step: dimensionally split, HLLC solver, parabolic reconstruction
        _case("kh 1030x770 fp32 split", "advance", "kh", 1030, 770, "fp32", 10, split=1),
        _case("kh 1024 fp32 hllc", "advance", "kh", 1024, 1024, "fp32", 10, riemann="hllc"),
        _case("kh 1000x700 fp32 ppm", "advance", "kh", 1000, 700, "fp32", 10, recon="ppm"),
        # a parameter study: independent problems on uneven grids, one graph per run
        _case("ensemble 48 fp32", "ensemble", "quad", 512, 512, "fp32", 10, members=48),
        # a run that lives in host memory
        _case("kh 1024 fp32 host", "host", "kh", 1024, 1024, "fp32", 2),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["advance"] * 6 + ["loop", "host", "ensemble"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    budget = 6.0e7 if precision == "fp32" else 1.5e6  # zones x steps: no dearer than the largest listed case
    if kind == "ensemble":
        c = _case(None, kind, "quad", rng.choice([128, 256, 512] if precision == "fp32" else [64, 128, 256]), 0, precision,
                  1, members=rng.randint(3, 56 if precision == "fp32" else 20))
        c["steps"] = max(1, min(rng.randint(2, 12), int(budget / _zones(c))))
        return c
    problem = rng.choice(["kh", "kh", "sod", "sedov", "rt", "quad"]) if kind != "host" else "kh"
    top = 3000 if precision == "fp32" else 1100
    if kind != "advance":
        top = 1000
    nx, ny = size(40, top), size(40, top)
    steps = max(1, min(24, int(budget / (nx * ny))))
    learned = kind != "loop" and precision == "fp32" and rng.random() < 0.2
    split = 0 if learned or kind == "host" else int(rng.random() < 0.25)
    riemann = "hllc" if not learned and rng.random() < 0.25 else "two-shock"
    recon = "ppm" if not learned and rng.random() < 0.25 else "plm"
    return _case(None, kind, problem, nx, ny, precision, steps, split, riemann, recon, learned,
                 fresh=kind != "host" and problem != "kh")


# ---- initial states -------------------------------------------------------------------------------------------------
def _sides(problem):
    return {"kh": (PERIODIC,) * 4, "sod": (OUTFLOW, OUTFLOW, PERIODIC, PERIODIC), "sedov": (OUTFLOW,) * 4,
            "quad": (OUTFLOW,) * 4, "rt": (PERIODIC, PERIODIC, HYDROSTATIC, HYDROSTATIC)}[problem]


def _domain(problem):
    return (0.0, 1.0, 0.0, 3.0) if problem == "rt" else (0.0, 1.0, 0.0, 1.0)


def _grav(problem):
    return -1.0 if problem == "rt" else 0.0


def _initial(problem, nx, ny, seed):
    """Interior conserved state (4, ny, nx) in double on the GPU."""
    dev = DEVICE
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    r = np.random.default_rng(int(seed))
    x0, x1, y0, y1 = _domain(problem)
    x = (x0 + (torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) * ((x1 - x0) / nx))[None, :].expand(ny, nx)
    y = (y0 + (torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) * ((y1 - y0) / ny))[:, None].expand(ny, nx)

    def noise():
        return 2.0 * torch.rand((ny, nx), dtype=torch.float64, device=dev, generator=g) - 1.0

    u = v = torch.zeros((), dtype=torch.float64, device=dev).expand(ny, nx)
    if problem == "kh":
        inner = (y - 0.5).abs() < 0.25
        rho, u = torch.where(inner, 2.0, 1.0), torch.where(inner, 0.5, -0.5)
        v = 0.01 * torch.sin(4.0 * math.pi * x) * noise()
        p = torch.full_like(rho, 2.5)
    elif problem == "sod":
        left = x < 0.5
        rl, pl, rr, pr = r.uniform(0.9, 1.1), r.uniform(0.9, 1.1), r.uniform(0.11, 0.14), r.uniform(0.09, 0.11)
        rho, p = torch.where(left, rl, rr), torch.where(left, pl, pr)
    elif problem == "sedov":
        rho = 1.0 + 0.01 * noise()
        r0 = max(0.01, 1.5 / min(nx, ny))
        p = torch.where((x - 0.5) ** 2 + (y - 0.5) ** 2 <= r0 ** 2, (GAMMA - 1.0) / (math.pi * r0 ** 2), 1e-5)
    elif problem == "rt":
        below = y < 1.5
        rho = torch.where(below, 1.0, 2.0)
        p = torch.where(below, 5.0 - y, 5.0 - 1.5 - 2.0 * (y - 1.5))
        v = 0.01 * torch.exp(-((y - 1.5) ** 2) / 0.1 ** 2) * (
            torch.cos(2.0 * math.pi * x) + r.uniform(0.1, 0.5) * torch.cos(4.0 * math.pi * (x + r.uniform())))
    else:
        q = (x >= 0.5).long() + 2 * (y >= 0.5).long()
        draw4 = lambda f: torch.tensor([f() for _ in range(4)], dtype=torch.float64, device=dev)[q]  # noqa: E731
        rho = draw4(lambda: math.exp(r.uniform(math.log(0.1), 0.0)))
        p = draw4(lambda: math.exp(r.uniform(math.log(0.01), math.log(10.0))))
        u, v = draw4(lambda: r.uniform(-1.0, 1.0)), draw4(lambda: r.uniform(-1.0, 1.0))
    rho, p = rho.double(), p.double()
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])


def _padded(U):
    P = torch.zeros((4, U.shape[1] + 2 * NG, U.shape[2] + 2 * NG), dtype=U.dtype, device=U.device)
    P[:, NG:-NG, NG:-NG] = U
    return P


def _dtype(case):
    return torch.float32 if case["precision"] == "fp32" else torch.float64


def _params(case, nx, ny):
    problem = case["problem"]
    x0, x1, y0, y1 = _domain(problem)
    return H.default_params(nx, ny, H.HYDRO_FP32 if case["precision"] == "fp32" else H.HYDRO_FP64, bc=_sides(problem),
                            gamma=GAMMA, cfl=CFL, xmin=x0, xmax=x1, ymin=y0, ymax=y1, grav=_grav(problem),
                            split=case["split"], riemann_solver=case["riemann"], reconstruction=case["recon"],
                            use_learned_guess=int(case["learned"]))


def _member_sizes(case, seed):
    sizes = [s for s in MEMBER_SIZES if s <= case["nx"]]
    # the sizes belong to the case, the states to the seed
    return [int(sizes[k]) for k in np.random.default_rng(case["members"]).integers(0, len(sizes), case["members"])]


def _member(case, k, n, seed):
    return _initial("quad", n, n, 1000003 * int(seed) + k)


def _trained_model(seed):
    """A network trained for a short while on faces over the range the step meets, their star pressures in 64 bits."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    r = torch.rand((6, 1 << 16), dtype=torch.float64, device="cuda", generator=g)
    a = [torch.exp(-2.0 * r[0]), 2.0 * r[1] - 1.0, torch.zeros_like(r[0]), torch.exp(6.0 * r[2] - 4.0)]
    b = [torch.exp(-2.0 * r[3]), 2.0 * r[4] - 1.0, torch.zeros_like(r[0]), torch.exp(6.0 * r[5] - 4.0)]
    star = _star_pressure(a, b)[0]
    m = Model(seed=int(seed))
    m.train(torch.stack([a[0], a[1], a[3], b[0], b[1], b[3], star, torch.ones_like(star)], dim=1).float().contiguous(),
            500, batch=4096, lr=3e-3, seed=1)
    return m


# ---- state and pass -------------------------------------------------------------------------------------------------
def prepare(case, seed):
    st = {"case": case, "turn": 0}
    if case["learned"]:
        st["model"] = _trained_model(seed)
    if case["kind"] == "ensemble":
        sizes = _member_sizes(case, seed)
        params = [_params(case, n, n) for n in sizes]
        st["ensemble"] = Ensemble(params, [_padded(_member(case, k, n, seed)).cpu().numpy() for k, n in enumerate(sizes)])
        st["ensemble"].autotune()
        return st
    nx, ny = case["nx"], case["ny"]
    U = _padded(_initial(case["problem"], nx, ny, seed)).to(_dtype(case))
    s = st["solver"] = Solver(_params(case, nx, ny))
    if case["learned"]:
        H.hydro_set_riemann_model(s.ctx, st["model"].m)
    if case["kind"] == "host":
        st["host"] = [U.cpu().pin_memory(), torch.zeros(U.shape, dtype=U.dtype).pin_memory()]
    elif case["fresh"]:
        st["host"] = U.cpu().pin_memory()
    else:
        s.current()[:, :, :s.NX].copy_(U)
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "ensemble":
        e = st["ensemble"]
        e.run(case["steps"])
        out = []
        for i, (NY, NX, pitch, _) in enumerate(e.shapes):
            buf = e.bufs[i][0 if H.hydro_batch_state(e.b, i) == e.bufs[i][0].data_ptr() else 1]
            out.append(buf.view(4, NY, pitch)[:, NG:NY - NG, NG:NX - NG])
        return out
    s = st["solver"]
    if case["kind"] == "host":
        for _ in range(case["steps"]):
            t = st["turn"]
            s.step_host(st["host"][t], st["host"][1 - t], chained=True)
            st["turn"] = 1 - t
        return st["host"][st["turn"]][:, NG:-NG, NG:-NG]
    if case["fresh"]:
        s.upload(st["host"])
    dts = []
    if case["kind"] == "loop":
        for _ in range(case["steps"]):
            s.fill_ghost()
            dts.append(s.cfl_dt())
            s.step(dts[-1])
    else:
        s.advance(case["steps"])
    state = s.current()[:, NG:-NG, NG:NG + case["nx"]]
    return {"state": state, "dt": dts} if dts else state


def _zones(case):
    if case["kind"] == "ensemble":
        return sum(n * n for n in _member_sizes(case, 0))
    return case["nx"] * case["ny"]


def work(case):
    # operations of the method per zone and step (the instrumented 64-bit count of the unsplit two-shock step, the
    # other forms from what they add or leave out); the state read and written once per pass
    flops = 1334 if case["precision"] == "fp64" else 1133
    if case["riemann"] == "hllc":
        flops -= 320
    if case["recon"] == "ppm":
        flops += 260
    if case["split"]:
        flops = 0.6 * flops
    zones = _zones(case)
    passes = case["steps"] if case["kind"] == "host" else 1
    return {"bytes": 2 * 4 * zones * (4 if case["precision"] == "fp32" else 8) * passes,
            "flops": flops * zones * case["steps"]}


# ---- the same steps in 64 bits, plain torch -------------------------------------------------------------------------
SMALL_DENS, SMALL_PRES, CVISC = 1e-10, 1e-20, 0.1


def exact(case, seed):
    if case["kind"] == "ensemble":
        out = []
        for k, n in enumerate(_member_sizes(case, seed)):
            U = _member(case, k, n, seed).to(_dtype(case)).double()
            out.append(_march(case, "quad", U)[0])
        return out
    U = _initial(case["problem"], case["nx"], case["ny"], seed).to(_dtype(case)).double()
    U, dts = _march(case, case["problem"], U)
    if case["kind"] == "host":
        return U.cpu()
    return {"state": U, "dt": dts} if case["kind"] == "loop" else U


def _march(case, problem, U):
    x0, x1, y0, y1 = _domain(problem)
    dx, dy = (x1 - x0) / U.shape[2], (y1 - y0) / U.shape[1]
    dts = []
    for k in range(case["steps"]):
        rho, u, v, p = _primitive(U)
        c = torch.sqrt(GAMMA * p / rho)
        dt = CFL * float(torch.minimum(dx / (u.abs() + c), dy / (v.abs() + c)).min())
        dts.append(dt)
        if case["split"]:
            for d in ((0, 1) if k % 2 == 0 else (1, 0)):
                U = _in_bands(_fill(U, problem, dy), lambda P: _sweep(case, P, d, dt, (dx, dy)[d], _grav(problem)))
        else:
            U = _in_bands(_fill(U, problem, dy), lambda P: _unsplit(case, P, dt, dx, dy, _grav(problem)))
    return U, dts


def _in_bands(P, step, rows=1024):
    """The step of a padded state, in bands of rows (a band's arrays are all that is held at once)."""
    ny = P.shape[1] - 2 * NG
    return torch.cat([step(P[:, j:min(j + rows, ny) + 2 * NG]) for j in range(0, ny, rows)], dim=1)


def _fill(U, problem, dy):
    """Padded state: periodic, zero-gradient and hydrostatic sides."""
    xs, _, ys, _ = _sides(problem)

    def index(n, side):
        i = torch.arange(-NG, n + NG, device=U.device)
        return i % n if side == PERIODIC else i.clamp(0, n - 1)

    ny = U.shape[1]
    P = U[:, index(ny, ys)][:, :, index(U.shape[2], xs)].clone()
    if ys == HYDROSTATIC:
        far = (torch.arange(-NG, ny + NG, device=U.device) - index(ny, ys)).double()[:, None]
        ke = 0.5 * (P[1] ** 2 + P[2] ** 2) / P[0]
        filled = ((GAMMA - 1.0) * (P[3] - ke) + P[0] * _grav(problem) * far * dy) / (GAMMA - 1.0) + ke
        P[3] = torch.where(far != 0, filled, P[3])
    return P


def _primitive(U):
    rho = U[0].clamp_min(SMALL_DENS)
    u, v = U[1] / rho, U[2] / rho
    return [rho, u, v, ((GAMMA - 1.0) * (U[3] - 0.5 * rho * (u * u + v * v))).clamp_min(SMALL_PRES)]


def _conserved(q):
    rho, u, v, p = q
    return [rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)]


def _at(a, k, d):
    """a[i + k] along direction d (0: x, the last axis; 1: y)."""
    return torch.roll(a, -k, -1 - d) if k else a


def _flattening(un, p, d):
    dp = _at(p, 1, d) - _at(p, -1, d)
    shock = (_at(un, -1, d) > _at(un, 1, d)) & (dp.abs() > 0.33 * torch.minimum(_at(p, 1, d), _at(p, -1, d)))
    z = dp.abs() / (_at(p, 2, d) - _at(p, -2, d)).abs().clamp_min(SMALL_PRES)
    chi = torch.where(shock, (1.0 - (z - 0.75) / 0.1).clamp(0.0, 1.0), 1.0)
    return torch.minimum(chi, torch.where(dp >= 0, _at(chi, -1, d), _at(chi, 1, d)))


def _mc(a, d):
    lo, hi = a - _at(a, -1, d), _at(a, 1, d) - a
    c = 0.5 * (lo + hi)
    s = torch.minimum(c.abs(), 2.0 * torch.minimum(lo.abs(), hi.abs()))
    return torch.where(lo * hi > 0, torch.where(c >= 0, s, -s), 0.0)


def _slope4(a, d):
    lo, hi = a - _at(a, -1, d), _at(a, 1, d) - a
    m = _mc(a, d)
    c = (4.0 / 3.0) * 0.5 * (lo + hi) - (_at(m, 1, d) + _at(m, -1, d)) / 6.0
    s = torch.minimum(c.abs(), 2.0 * torch.minimum(lo.abs(), hi.abs()))
    return torch.where(lo * hi > 0, torch.where(c >= 0, s, -s), 0.0)


def _waves(q):
    """Sound speed and the projections of a jump on the acoustic (-, +) and entropy waves of q = (rho, un, ut, p)."""
    c = torch.sqrt(GAMMA * q[3] / q[0])
    minus = lambda j: -0.5 * q[0] / c * j[1] + 0.5 * j[3] / c ** 2  # noqa: E731
    plus = lambda j: 0.5 * q[0] / c * j[1] + 0.5 * j[3] / c ** 2  # noqa: E731
    entropy = lambda j: j[0] - j[3] / c ** 2  # noqa: E731
    return c, minus, plus, entropy


def _add_wave(o, q, c, minus=None, plus=None, entropy=None, shear=None):
    if minus is not None:
        o[0], o[1], o[3] = o[0] + minus, o[1] - minus * c / q[0], o[3] + minus * c * c
    if plus is not None:
        o[0], o[1], o[3] = o[0] + plus, o[1] + plus * c / q[0], o[3] + plus * c * c
    if entropy is not None:
        o[0], o[2] = o[0] + entropy, o[2] + shear
    return o


def _trace(case, q, xi, sigma, d):
    """Half-step states of each cell's far (+) and near (-) face, q = (rho, un, ut, p)."""
    c, minus, plus, entropy = _waves(q)
    un = q[1]
    zero = torch.zeros_like(un)
    on = lambda m, a: torch.where(m, a, zero)  # noqa: E731
    if case["recon"] == "plm":
        dq = [xi * _slope4(a, d) for a in q]
        h = 0.5 * sigma
        far = [a + 0.5 * (1.0 - sigma * (un + c)) * s for a, s in zip(q, dq)]
        far = _add_wave(far, q, c, minus=on(un - c >= 0, h * 2.0 * c * minus(dq)),
                        entropy=on(un >= 0, h * c * entropy(dq)), shear=on(un >= 0, h * c * dq[2]))
        near = [a - 0.5 * (1.0 + sigma * (un - c)) * s for a, s in zip(q, dq)]
        near = _add_wave(near, q, c, plus=on(un + c <= 0, -h * 2.0 * c * plus(dq)),
                         entropy=on(un <= 0, -h * c * entropy(dq)), shear=on(un <= 0, -h * c * dq[2]))
    else:
        lo, hi = [], []
        for a in q:
            m = _mc(a, d)
            e = a + 0.5 * (_at(a, 1, d) - a) - (_at(m, 1, d) - m) / 6.0
            l, r = _at(e, -1, d), e
            flat = (r - a) * (a - l) <= 0
            w, mid = r - l, a - 0.5 * (l + r)
            left = w * mid > w * w / 6.0
            right = ~left & (-(w * w) / 6.0 > w * mid)
            l2 = torch.where(flat, a, torch.where(left, 3.0 * a - 2.0 * r, l))
            r2 = torch.where(flat, a, torch.where(right, 3.0 * a - 2.0 * l, r))
            lo.append(xi * l2 + (1.0 - xi) * a)
            hi.append(xi * r2 + (1.0 - xi) * a)
        w = [r - l for l, r in zip(lo, hi)]
        a6 = [6.0 * (a - 0.5 * (l + r)) for a, l, r in zip(q, lo, hi)]

        def mean(s, side):  # average over the fraction s of the cell next to a face
            if side > 0:
                return [r - 0.5 * s * (j - (1.0 - 2.0 / 3.0 * s) * k) for r, j, k in zip(hi, w, a6)]
            return [l + 0.5 * s * (j + (1.0 - 2.0 / 3.0 * s) * k) for l, j, k in zip(lo, w, a6)]

        def side_state(side):
            speeds = [sigma * side * s for s in (un - c, un, un + c)]
            ref = mean(speeds[2 if side > 0 else 0].clamp_min(0.0), side)
            off = [[a - b for a, b in zip(ref, mean(s, side))] for s in speeds]
            m = [s >= 0 for s in speeds]
            return _add_wave(list(ref), q, c, minus=on(m[0], -minus(off[0])), plus=on(m[2], -plus(off[2])),
                             entropy=on(m[1], -entropy(off[1])), shear=on(m[1], -off[1][2]))

        far, near = side_state(1), side_state(-1)
    for o in (far, near):
        o[0], o[3] = o[0].clamp_min(SMALL_DENS), o[3].clamp_min(SMALL_PRES)
    return far, near


def _star_pressure(a, b):
    """Two-shock star pressure and mass fluxes of the faces between a and b = (rho, un, ut, p)."""
    g1 = (GAMMA + 1.0) / (2.0 * GAMMA)
    ca, cb = torch.sqrt(GAMMA * a[3] * a[0]), torch.sqrt(GAMMA * b[3] * b[0])
    scale = a[1].abs() + b[1].abs() + ca / a[0] + cb / b[0]
    flux = lambda p, q, c: c * torch.sqrt(1.0 + g1 * (p / q[3] - 1.0))  # noqa: E731
    p = ((cb * a[3] + ca * b[3] + ca * cb * (a[1] - b[1])) / (ca + cb)).clamp_min(SMALL_PRES)
    for _ in range(32):
        wa, wb = flux(p, a, ca), flux(p, b, cb)
        za, zb = 2.0 * wa ** 3 / (wa * wa + ca * ca), 2.0 * wb ** 3 / (wb * wb + cb * cb)
        new = (p - za * zb * (b[1] + (p - b[3]) / wb - a[1] + (p - a[3]) / wa) / (za + zb)).clamp_min(SMALL_PRES)
        step = (new - p).abs()
        p = new
        if bool(((step <= 1e-14 * p) | (step * (za + zb) / (za * zb) <= 1e-14 * scale)).all()):
            break
    return p, flux(p, a, ca), flux(p, b, cb)


def _flux(q):
    rho, u, v, p = q
    return [rho * u, rho * u * u + p, rho * u * v, u * (p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v) + p)]


def _riemann(case, a, b):
    """Flux through the faces between the states a (below or left) and b."""
    if case["riemann"] == "hllc":
        ca, cb = torch.sqrt(GAMMA * a[3] / a[0]), torch.sqrt(GAMMA * b[3] / b[0])
        sa, sb = torch.minimum(a[1] - ca, b[1] - cb), torch.maximum(a[1] + ca, b[1] + cb)
        ma, mb = a[0] * (sa - a[1]), b[0] * (sb - b[1])
        s = (b[3] - a[3] + ma * a[1] - mb * b[1]) / (ma - mb)
        left = (sa >= 0) | (s >= 0)
        o = [torch.where(left, x, y) for x, y in zip(a, b)]
        so = torch.where(left, sa, sb)
        jump = torch.where(left, sa < 0, sb >= 0)
        U, F = _conserved(o), _flux(o)
        f = o[0] * (so - o[1]) / (so - s)
        star = [f, f * s, f * o[2], f * (U[3] / o[0] + (s - o[1]) * (s + o[3] / (o[0] * (so - o[1]))))]
        return [torch.where(jump, x + so * (y - z), x) for x, y, z in zip(F, star, U)]
    p, wa, wb = _star_pressure(a, b)
    u = (wa * a[1] + wb * b[1] + (a[3] - b[3])) / (wa + wb)
    left = u > 0
    sign = torch.where(left, 1.0, -1.0).double()
    o = [torch.where(left, x, y) for x, y in zip(a, b)]
    w = torch.where(left, wa, wb)
    rho = 1.0 / (1.0 / o[0] - (p - o[3]) / (w * w))
    shock = p > o[3]
    head = torch.where(shock, o[1] - sign * w / o[0], o[1] - sign * torch.sqrt(GAMMA * o[3] / o[0]))
    tail = u - sign * torch.sqrt(GAMMA * p / rho)
    outside, inside = sign * head >= 0, shock | (sign * tail <= 0)
    frac = torch.where(outside, 0.0, torch.where(inside, 1.0, head / (head - tail)))
    still = u == 0
    state = [torch.where(still, 0.5 * (a[0] + b[0]), torch.where(inside & ~outside, rho, o[0] + frac * (rho - o[0]))),
             torch.where(inside & ~outside | still, u, o[1] + frac * (u - o[1])),
             torch.where(still, 0.5 * (a[2] + b[2]), o[2]),
             torch.where(inside & ~outside | still, p, o[3] + frac * (p - o[3]))]
    return _flux(state)


def _frame(q, d):
    return q if d == 0 else [q[0], q[2], q[1], q[3]]


def _faces(case, far, near, d):
    """Flux through each cell's face at its + side, in (rho, x, y, E) order; far and near in the face frame."""
    return _frame(_riemann(case, far, [_at(a, 1, d) for a in near]), d)


def _viscosity(P, F, rate, d):
    """F with the artificial viscosity of its + face, rate = -(divergence x spacing)."""
    av = CVISC * rate.clamp_min(0.0)
    return [f + av * (U - _at(U, 1, d)) for f, U in zip(F, P)]


def _interior(U):
    return torch.stack([a[NG:-NG, NG:-NG] for a in U])


def _gravity_sources(P, U, dt, grav):
    if grav:
        U[2] = U[2] + 0.5 * dt * grav * (P[0] + U[0])
        U[3] = U[3] + 0.5 * dt * grav * (P[2] + U[2])
    return U


def _unsplit(case, P, dt, dx, dy, grav):
    P = list(P)
    q = _primitive(P)
    u, v = q[1], q[2]
    h = (dx, dy)
    xi = torch.minimum(_flattening(u, q[3], 0), _flattening(v, q[3], 1))
    traced = []
    for d in (0, 1):
        states = _trace(case, _frame(q, d), xi, dt / h[d], d)
        for s in states:
            s[2 - d] = s[2 - d] + 0.5 * dt * grav
        traced.append(states)
    hat = [_faces(case, *traced[d], d) for d in (0, 1)]
    F = []
    for d in (0, 1):
        t = 1 - d
        change = [0.5 * dt / h[t] * (f - _at(f, -1, t)) for f in hat[t]]
        far, near = [_frame(_primitive([a - b for a, b in zip(_conserved(_frame(s, d)), change)]), d) for s in traced[d]]
        un, ut = (u, v) if d == 0 else (v, u)
        across = _at(ut, 1, t) - _at(ut, -1, t)
        div = (_at(un, 1, d) - un) / h[d] + (_at(across, 1, d) + across) / (4.0 * h[t])
        F.append(_viscosity(P, _faces(case, far, near, d), -div * h[d], d))
    U = [a + dt / dx * (_at(f, -1, 0) - f) + dt / dy * (_at(g, -1, 1) - g) for a, f, g in zip(P, *F)]
    return _interior(_gravity_sources(P, U, dt, grav))


def _sweep(case, P, d, dt, h, grav):
    P = list(P)
    q = _frame(_primitive(P), d)
    far, near = _trace(case, q, _flattening(q[1], q[3], d), dt / h, d)
    for s in (far, near):
        s[2 - d] = s[2 - d] + 0.5 * dt * grav
    F = _viscosity(P, _faces(case, far, near, d), q[1] - _at(q[1], 1, d), d)
    U = [a + dt / h * (_at(f, -1, d) - f) for a, f in zip(P, F)]
    return _interior(_gravity_sources(P, U, dt, grav if d == 1 else 0.0))
