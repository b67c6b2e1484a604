"""Timing cases of the library: the calls a simulation program makes, over the range of sizes,
dimensions, precisions and options that the workloads of this repository cover.

A case names a workload family (``family``), its grid, the compute form (``form``: "mixed" or
"fp64") and the call it times (``call``):

* ``step``   one ``es_step`` of a time loop (mesh redistribution + SSP-RK3 step, in place);
* ``batch``  one ``es_step_batch`` over independent instances of uneven grids;
* ``host``   one ``es_run_host`` step on pinned host buffers (the copies included);
* ``diag``   what an output step runs: ``es_rhs``, ``entropy_production``, ``es_schlieren``.

``listed()`` gives the fixed cases and ``draw(rng)`` random ones of the same ranges;
``prepare(case, seed)`` builds the inputs from the seed, ``run(state)`` makes one pass and
returns its outputs, ``work(case)`` counts the bytes and flops a pass cannot do without, and
``exact(case, seed)`` evaluates the same pass in binary64 with plain torch operations.
"""
import math
import random

import numpy as np
import torch

from paper_2202_07989_gb300 import es as ES
from paper_2202_07989_gb300 import workloads as W


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # the isentropic vortex of the accuracy study (Example 5.1), 64^2 periodic, adaptive mesh
        # with the default ten sweeps: the smallest steps, where launches and latency count
        {"name": "step_vortex_64_mixed", "call": "step", "family": "vortex", "n0": 64, "n1": 64, "form": "mixed"},
        # the same problem with its prescribed mesh motion, FP64: residual, entropy production and
        # schlieren field, as an accuracy study or an output step evaluates them
        {"name": "diag_vortex_64_fp64", "call": "diag", "family": "vortex", "n0": 64, "n1": 64, "form": "fp64"},
        # the benchmark's headline: the 2D two-component shock-bubble on 400 x 200, tuned
        {"name": "step_bubble_400x200_mixed", "call": "step", "family": "bubble", "n0": 400, "n1": 200, "form": "mixed",
         "tune": True},
        # the same step in the FP64 form (the reference form of every accuracy statement)
        {"name": "step_bubble_400x200_fp64", "call": "step", "family": "bubble", "n0": 400, "n1": 200, "form": "fp64"},
        # WENO-JS on the 350 x 150 grid of the tri-point problem (the MM-WENOJS comparison runs);
        # neither extent is a multiple of a tile
        {"name": "step_bubble_350x150_js", "call": "step", "family": "bubble", "n0": 350, "n1": 150, "form": "mixed",
         "weno": 1},
        # the finest uniform-mesh run of the 2D shock-bubble, 2400 x 480 (UM-WENOMR)
        {"name": "step_bubble_2400x480_um", "call": "step", "family": "bubble", "n0": 2400, "n1": 480, "form": "mixed",
         "fixed": True},
        # one step per call on host buffers at the 800 x 160 grid of the shock-bubble runs: a host
        # program that couples the library to its own code
        {"name": "host_bubble_800x160_mixed", "call": "host", "family": "bubble", "n0": 800, "n1": 160, "form": "mixed"},
        # a parameter study: 32 independent instances of uneven square grids 96..512, tuned
        {"name": "batch_32_mixed", "call": "batch", "family": "batch", "count": 32, "nmin": 96, "nmax": 512,
         "sizes": 2202, "form": "mixed", "tune": True},
        # the 3D octant Riemann problem of the benchmark, 128^3, adaptive mesh
        {"name": "step_riemann3d_128_mixed", "call": "step", "family": "riemann", "n0": 128, "form": "mixed"},
        # the 3D two-component shock-bubble (Example 5.10 shape), 128 x 64 x 64, adaptive mesh
        {"name": "step_bubble3d_64_mixed", "call": "step", "family": "bubble3d", "n0": 64, "form": "mixed"},
        # the stiffened-gas 3D shock-bubble (Example 5.11) on 400 x 80 x 80, uniform mesh
        {"name": "step_stiffened_80_um", "call": "step", "family": "stiffened", "n0": 80, "form": "mixed", "fixed": True},
        # the 3D Riemann problem in the FP64 form, on an odd grid
        {"name": "step_riemann3d_63_fp64", "call": "step", "family": "riemann", "n0": 63, "form": "fp64"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges (no name); sizes log-uniform, odd ones among them."""
    form = "mixed" if rng.random() < 0.75 else "fp64"
    kind = rng.choice(["2d", "2d", "2d", "3d", "3d", "batch", "host", "diag"])
    if kind == "batch":
        return {"call": "batch", "family": "batch", "count": rng.randint(2, 24), "nmin": 48,
                "nmax": rng.randint(96, 320 if form == "mixed" else 128), "sizes": rng.randrange(1 << 20), "form": form}
    if kind == "3d":
        fam = rng.choice(["riemann", "bubble3d", "stiffened"])
        hi = {"riemann": 112, "bubble3d": 64, "stiffened": 64}[fam] if form == "mixed" else \
             {"riemann": 56, "bubble3d": 36, "stiffened": 28}[fam]
        c = {"call": "step", "family": fam, "n0": _logint(rng, 16, hi), "form": form}
        if fam == "stiffened" or rng.random() < 0.2:
            c["fixed"] = True
        return c
    if kind == "diag":
        fam = rng.choice(["vortex", "bubble"])
        n0 = _logint(rng, 48, 800)
        n1 = n0 if fam == "vortex" else _logint(rng, 40, 200)
        if fam == "vortex":
            n0 = n1 = min(n0, 300)
        return {"call": "diag", "family": fam, "n0": n0, "n1": n1, "form": form}
    fam = rng.choice(["vortex", "bubble", "bubble"])
    n0 = _logint(rng, 48, 1200 if form == "mixed" else 500)
    n1 = n0 if fam == "vortex" else _logint(rng, 40, 480 if form == "mixed" else 240)
    if fam == "vortex":
        n0 = n1 = min(n0, 512 if form == "mixed" else 256)
    c = {"call": "host" if kind == "host" else "step", "family": fam, "n0": n0, "n1": n1, "form": form}
    if fam == "bubble":
        if rng.random() < 0.25:
            c["weno"] = 1
        if rng.random() < 0.25:
            c["fixed"] = True
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _batch_sizes(case):
    r = random.Random(int(case["sizes"]))
    return [r.randint(int(case["nmin"]), int(case["nmax"])) for _ in range(int(case["count"]))]


def _shape(case):
    """(d, N, [(n0, n1, n2), ...]) of the case's instances."""
    fam, n = case["family"], int(case.get("n0", 0))
    if fam == "batch":
        return 2, 2, [(m, m, 1) for m in _batch_sizes(case)]
    if fam in ("vortex", "bubble"):
        return 2, 1 if fam == "vortex" else 2, [(n, int(case["n1"]), 1)]
    return 3, 1 if fam == "riemann" else 2, [{"riemann": (n, n, n), "bubble3d": (2 * n, n, n), "stiffened": (5 * n, n, n)}[fam]]


def _roughen(pb, U, x, rng, state=0.02):
    """The initial data of a workload as a run in progress holds it: densities, momenta and energy
    varied smoothly by about 2% (no region stays exactly constant) and, on a moving mesh, the nodes
    displaced smoothly by a fraction of a cell."""
    f = np.zeros(pb.shape)
    xi = W.xi_nodes(pb)
    for _ in range(3):
        term = np.full(pb.shape, rng.uniform(-1, 1))
        for k in range(pb.d):
            term = term * np.cos(2 * math.pi * rng.integers(1, 4) * (xi[k] - pb.xi_lo[k]) / pb.length[k] + rng.uniform(0, 2 * math.pi))
        f += term
    if not pb.fixed_mesh:
        x = x + (W.smooth_mesh(pb, rng, amp=0.05) - np.stack(xi))
    return U * (1.0 + state * f), x


def _problems(case, seed):
    """[(problem, U, x, xdot or None)] of the case, from the seed alone."""
    rng = np.random.default_rng(int(seed))
    fam, fixed, weno = case["family"], bool(case.get("fixed")), int(case.get("weno", 0))
    out = []
    if fam == "vortex":
        pb, U, x, xdot = W.vortex_2d(int(case["n0"]), t=float(rng.uniform(0.0, 6.0)))
        out.append((pb, U, x, xdot))
    elif fam == "bubble":
        pb, U, x = W.shock_bubble_2d(int(case["n0"]), int(case["n1"]), Ms=float(rng.uniform(1.15, 1.3)),
                                     radius=float(rng.uniform(0.17, 0.23)), mu=5)
        out.append((pb, U, x, None))
    elif fam == "riemann":
        pb, U, x = W.riemann_3d(int(case["n0"]), seed=int(rng.integers(1 << 30)))
        out.append((pb, U, x, None))
    elif fam == "bubble3d":
        pb, U, x = W.shock_bubble_3d(int(case["n0"]), Ms=float(rng.uniform(1.15, 1.3)), radius=float(rng.uniform(0.18, 0.22)))
        out.append((pb, U, x, None))
    elif fam == "stiffened":
        pb, U, x = W.shock_bubble_3d_stiffened(int(case["n0"]), Ms=float(rng.uniform(9.0, 10.0)))
        out.append((pb, U, x, None))
    else:
        for n in _batch_sizes(case):
            # the bubble kept clear of the shock at x_1 = 0.8 (a bubble that touches it goes
            # non-physical in the first step)
            prm = dict(n=n, Ms=float(rng.uniform(1.1, 3.0)), r=float(rng.uniform(0.1, 0.27)),
                       g2=float(rng.uniform(1.1, 4.4)), pi2=float(rng.uniform(0.0, 10.0)))
            pb, U, x = W.batched_instance(prm)
            out.append((pb, U, x, None))
    done = []
    for pb, U, x, xdot in out:
        pb = pb.with_(weno=weno, fixed_mesh=fixed or pb.fixed_mesh)
        if fam != "vortex":
            U, x = _roughen(pb, U, x, rng, state=0.005 if fam in ("stiffened", "batch") else 0.02)
        done.append((pb, U, x, xdot))
    return done


class _State:
    pass


def _initial(case, seed):
    """[(problem, JU, J, x, xdot or None)] and the flat block that holds every (JU | J | x), as a
    program that checkpoints its state with one copy keeps it."""
    probs = _problems(case, seed)
    flat = torch.empty(sum((pb.nc + 1 + pb.d) * pb.ncell for pb, _, _, _ in probs), dtype=torch.float64, device="cuda")
    out, at = [], 0
    for pb, U, x, xdot in probs:
        blk = flat[at: at + (pb.nc + 1 + pb.d) * pb.ncell].view((pb.nc + 1 + pb.d,) + pb.shape)
        at += blk.numel()
        JU, J, xg = blk[: pb.nc], blk[pb.nc], blk[pb.nc + 1:]
        xg.copy_(torch.from_numpy(np.ascontiguousarray(x)))
        J.copy_(_det_J(pb, xg))
        JU.copy_(torch.from_numpy(np.ascontiguousarray(U)))
        JU *= J
        out.append((pb, JU, J, xg, None if xdot is None else torch.from_numpy(np.ascontiguousarray(xdot)).cuda()))
    return out, flat


def prepare(case, seed):
    s = _State()
    s.call = case["call"]
    form = ES.MIXED if case["form"] == "mixed" else ES.FP64
    inst, s.flat = _initial(case, seed)
    pb, s.JU, s.J, s.x, xdot = inst[0]
    if s.call == "batch":
        # one block for the states, one for the velocities, one for the time steps of all instances
        s.ctx = ES.es_create_batch([p for p, _, _, _, _ in inst], form)
        s.xdots = torch.zeros(sum(x.numel() for _, _, _, x, _ in inst), dtype=torch.float64, device="cuda")
        s.dts = torch.zeros((len(inst), 2), dtype=torch.float64, device="cuda")
        xdots = [v.view_as(x) for v, (_, _, _, x, _) in zip(s.xdots.split([x.numel() for _, _, _, x, _ in inst]), inst)]
        s.ctx.es_bind_batch([i[1] for i in inst], [i[2] for i in inst], [i[3] for i in inst], xdots, list(s.dts))
        if case.get("tune"):
            s.ctx.es_autotune()
        return s
    s.ctx = ES.es_create(pb, form)
    if s.call == "host":
        h = torch.empty((pb.nc + 1 + pb.d,) + pb.shape, dtype=torch.float64, pin_memory=True)
        h.copy_(s.flat.view_as(h))
        s.JU, s.J, s.x = h[: pb.nc], h[pb.nc], h[pb.nc + 1:]
        return s
    if s.call == "diag":
        s.xdot = xdot if xdot is not None else torch.zeros_like(s.x)
        s.dJU, s.dJ = torch.empty_like(s.JU), torch.empty_like(s.J)
        s.ent = torch.empty(2, dtype=torch.float64, device="cuda")
        s.phi = torch.empty_like(s.J)
    else:
        s.xdot = torch.zeros_like(s.x)
        s.dt = torch.zeros(2, dtype=torch.float64, device="cuda")
        if case.get("tune"):
            s.ctx.es_autotune(s.JU, s.J, s.x)
    return s


def run(s):
    if s.call == "step":
        s.ctx.es_step(s.JU, s.J, s.x, xdot=s.xdot, dt_dtau=s.dt)
        return {"JU": s.JU, "J": s.J, "x": s.x, "xdot": s.xdot, "dt": s.dt}
    if s.call == "batch":
        s.ctx.es_step_batch()
        return {"state": s.flat, "xdot": s.xdots, "dt": s.dts}
    if s.call == "host":
        t = s.ctx.es_run_host(s.JU, s.J, s.x, 1)
        return {"JU": s.JU, "J": s.J, "x": s.x, "t": t}
    s.ctx.es_rhs(s.JU, s.J, s.x, s.xdot, dJU=s.dJU, dJ=s.dJ)
    s.ctx.entropy_production(s.JU, s.J, s.dJU, s.dJ, out=s.ent)
    s.ctx.es_schlieren(s.JU, s.J, s.x, phi=s.phi)
    return {"dJU": s.dJU, "dJ": s.dJ, "entropy": s.ent, "phi": s.phi}


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    """Bytes: the state read and written once (and the fields a call returns).  Flops: per
    interface and stage three distinct two-point fluxes, the GCL stencil and, per characteristic
    column, the projection and two WENO evaluations; per node the metrics and, on a moving mesh,
    the monitor, filter and sweeps of a step."""
    d, N, sizes = _shape(case)
    nc = N + d + 1
    cells = sum(a * b * c for a, b, c in sizes)
    pair = 26 + 18 * d + 21 * N
    setup = (2 if d == 2 else 15) + 3 * d + 2 * d * d + (12 if N == 1 else 45) + 4
    iface = 3 * pair + 10 + 11 * d + setup + nc * (8 + 15 * nc + 2 * d * d + 192) + nc
    metrics = 24 if d == 2 else 200
    fixed = bool(case.get("fixed"))
    mu = 0 if fixed else (5 if case["family"] in ("bubble", "batch") else 10)
    mesh = 40 + (0 if fixed else 2 * d * 4 + 3 * 3 ** d * 2 + mu * (2 * d * (2 * d + 3) + d))
    state = 8 * (nc + 1 + d)
    if case["call"] == "diag":
        return {"bytes": float(cells * (state + 8 * d + 8 * (nc + 1) + 8)), "flops": float(cells * (d * iface + 2 * metrics + 60))}
    per = 3 * (d * iface + (nc + 1) * 4) + (1 if fixed else (2 if d == 2 else 3)) * metrics + mesh
    return {"bytes": float(cells * (2 * state + 8 * d)), "flops": float(cells * per)}


# --------------------------------------------------------------------------
# the same pass in binary64 with plain torch operations (the paper's formulas, field by field)
# --------------------------------------------------------------------------

_ALPHA = (1.5, -0.3, 1.0 / 30.0)


def _dim(k):
    return -1 - k           # direction k of an array (..., n3, n2, n1)


def _take(a, k, idx):
    return a.index_select(a.dim() + _dim(k), torch.tensor(idx, device=a.device))


def _sl(a, k, start, length):
    return a.narrow(a.dim() + _dim(k), start, length)


def _ext_x(pb, x, k, g, vel=False):
    """Positions (or velocities) with g ghost layers along k: wrap with the period, else mirror."""
    n = pb.n[k]
    lo, hi = pb.xi_lo[k], pb.xi_lo[k] + pb.length[k]
    if pb.bc[k][0] == W.PERIODIC:
        a, b = _take(x, k, [(i % n) for i in range(-g, 0)]).clone(), _take(x, k, [i % n for i in range(n, n + g)]).clone()
        if not vel:
            a[k] -= pb.length[k]
            b[k] += pb.length[k]
    else:
        a, b = _take(x, k, [-1 - i for i in range(-g, 0)]).clone(), _take(x, k, [2 * n - 1 - i for i in range(n, n + g)]).clone()
        a[k] = -a[k] if vel else 2 * lo - a[k]
        b[k] = -b[k] if vel else 2 * hi - b[k]
    return torch.cat([a, x, b], dim=x.dim() + _dim(k))


def _ext_U(pb, U, k, g):
    n, sides = pb.n[k], []
    for s in range(2):
        gh = list(range(-g, 0)) if s == 0 else list(range(n, n + g))
        kind = pb.bc[k][s]
        if kind == W.PERIODIC:
            e = _take(U, k, [i % n for i in gh])
        elif kind == W.REFLECT:
            e = _take(U, k, [(-1 - i) if s == 0 else (2 * n - 1 - i) for i in gh]).clone()
            e[pb.N + k] = -e[pb.N + k]
        elif kind == W.OUTFLOW:
            e = _take(U, k, [0 if s == 0 else n - 1 for _ in gh])
        else:
            e = _take(U, k, [0] * g).clone()
            for q in range(pb.nc):
                e[q] = float(pb.inflow[k, s, q])
        sides.append(e)
    return torch.cat([sides[0], U, sides[1]], dim=U.dim() + _dim(k))


def _ext_s(pb, a, k, g):
    n = pb.n[k]
    if pb.bc[k][0] == W.PERIODIC:
        lo, hi = [i % n for i in range(-g, 0)], [i % n for i in range(n, n + g)]
    else:
        lo, hi = [0] * g, [n - 1] * g
    return torch.cat([_take(a, k, lo), a, _take(a, k, hi)], dim=a.dim() + _dim(k))


def _delta(a, k):
    """delta_k[a] = 1/2 sum_m alpha_m (a_{+m} - a_{-m}); the array shrinks by 3 at both ends of k."""
    n = a.shape[a.dim() + _dim(k)] - 6
    return 0.5 * sum(_ALPHA[m - 1] * (_sl(a, k, 3 + m, n) - _sl(a, k, 3 - m, n)) for m in (1, 2, 3))


def _metrics_row(pb, x, k):
    """J xi_k/x_j, j = 1..d, with 3 ghost layers along k (interior in the other directions)."""
    if pb.d == 2:
        o = 1 - k
        e = _ext_x(pb, _ext_x(pb, x, k, 3), o, 3)
        dx = _delta(e, o) / pb.dxi[o]
        return [dx[1], -dx[0]] if k == 0 else [-dx[1], dx[0]]
    a, b = ((2, 1), (0, 2), (1, 0))[k]
    e = _ext_x(pb, _ext_x(pb, _ext_x(pb, x, k, 3), a, 3), b, 3)
    row = []
    for p, q in ((1, 2), (2, 0), (0, 1)):
        ca = _sl(e, a, 3, pb.n[a])
        cb = _sl(e, b, 3, pb.n[b])
        t = _delta(_delta(e[p], b) * cb[q], a) - _delta(_delta(e[p], a) * ca[q], b)
        row.append(t / (pb.dxi[a] * pb.dxi[b]))
    return row


def _det_J(pb, x):
    A = [[_delta(_ext_x(pb, x, k, 3), k)[j] / pb.dxi[k] for k in range(pb.d)] for j in range(pb.d)]
    if pb.d == 2:
        return A[0][0] * A[1][1] - A[0][1] * A[1][0]
    return (A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0])
            + A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]))


def _prim(pb, U):
    N, d = pb.N, pb.d
    rho = sum(U[l] for l in range(N))
    v = [U[N + m] / rho for m in range(d)]
    cvr = sum(pb.cv[l] * U[l] for l in range(N))
    rr = sum(pb.R(l) * U[l] for l in range(N))
    pinf = sum(pb.pinf[:N])
    T = (U[N + d] - 0.5 * rho * sum(m * m for m in v) - pinf) / cvr
    return rho, v, T, rr * T - pinf, rr / rho, sum(pb.gamma[l] * pb.cv[l] * U[l] for l in range(N)) / cvr


def _entropy_vars(pb, U, v, T):
    v2 = sum(m * m for m in v)
    V = [-(pb.cv[l] * torch.log(T) - pb.R(l) * torch.log(U[l])) - v2 / (2 * T) + pb.cv[l] * pb.gamma[l] for l in range(pb.N)]
    return torch.stack(V + [m / T for m in v] + [-1.0 / T])


def _lm(a, b):
    """Logarithmic mean, the Ismail-Roe series at small jumps."""
    f = (b - a) / (b + a)
    u = f * f
    small = u < 1e-4
    lr = torch.log(b) - torch.log(a)
    return torch.where(small, 0.5 * (a + b) / (1 + u / 3 + u * u / 5 + u * u * u / 7), (b - a) / torch.where(small, torch.ones_like(lr), lr))


def _pair(pb, A, B):
    """Two-point flux of node sets A and B: (rho_l, v, beta, [Mt, Mx...])."""
    N, d = pb.N, pb.d
    (ra, va, ba, ma), (rb, vb, bb, mb) = A, B
    lr = [_lm(ra[l], rb[l]) for l in range(N)]
    lb, ab = _lm(ba, bb), 0.5 * (ba + bb)
    vm = [0.5 * (va[m] + vb[m]) for m in range(d)]
    hv2 = sum(0.25 * (va[m] * va[m] + vb[m] * vb[m]) for m in range(d))
    M = [0.5 * (ma[c] + mb[c]) for c in range(d + 1)]
    pinf = sum(pb.pinf[:N])
    sr = sum(lr)
    P = sum(pb.R(l) * 0.5 * (ra[l] + rb[l]) for l in range(N)) / ab - pinf
    e = sum(lr[l] * (pb.cv[l] / lb - hv2) for l in range(N)) + sr * sum(m * m for m in vm)
    un = sum(M[1 + j] * vm[j] for j in range(d))
    ut = M[0] + un
    F = [ut * lr[l] for l in range(N)] + [ut * sr * vm[m] + M[1 + m] * P for m in range(d)]
    F.append(ut * e + pinf * M[0] + un * (P + pinf))
    return torch.stack(F)


def _weno_mr(pb, w):
    m2, m1, c, p1, p2 = w
    a2, a3 = 0.5 * (p1 - m1), 0.5 * (m1 - 2 * c + p1)
    b2 = (11 * m2 - 82 * m1 + 82 * p1 - 11 * p2) / 120
    b3 = (-3 * m2 + 40 * m1 - 74 * c + 40 * p1 - 3 * p2) / 56
    b4 = (-m2 + 2 * m1 - 2 * p1 + p2) / 12
    b5 = (m2 - 4 * m1 + 6 * c - 4 * p1 + p2) / 24
    be1 = torch.minimum((c - m1) ** 2, (p1 - c) ** 2)
    be2 = a2 * a2 + 13.0 / 3 * a3 * a3
    t1, t2 = b2 + b4 / 10, b3 + 123.0 / 455 * b5
    be3 = t1 * t1 + 13.0 / 3 * t2 * t2 + 781.0 / 20 * b4 * b4 + 1421461.0 / 2275 * b5 * b5
    tau = (0.5 * ((be3 - be1).abs() + (be3 - be2).abs())) ** 2
    x1, x2, x3 = pb.chi
    o = [x1 * (1 + tau / (pb.weno_eps + be1)), x2 * (1 + tau / (pb.weno_eps + be2)), x3 * (1 + tau / (pb.weno_eps + be3))]
    h2, h3 = c + a2 / 2 + a3 / 6, c + b2 / 2 + b3 / 6 + b4 / 20 + b5 / 70
    return (o[0] * c + o[1] * h2 + o[2] * (h3 / x3 - x1 / x3 * c - x2 / x3 * h2)) / (o[0] + o[1] + o[2])


def _weno_js(pb, w):
    m2, m1, c, p1, p2 = w
    q = [(2 * m2 - 7 * m1 + 11 * c) / 6, (-m1 + 5 * c + 2 * p1) / 6, (2 * c + 5 * p1 - p2) / 6]
    b = [13.0 / 12 * (m2 - 2 * m1 + c) ** 2 + 0.25 * (m2 - 4 * m1 + 3 * c) ** 2,
         13.0 / 12 * (m1 - 2 * c + p1) ** 2 + 0.25 * (m1 - p1) ** 2,
         13.0 / 12 * (c - 2 * p1 + p2) ** 2 + 0.25 * (3 * c - 4 * p1 + p2) ** 2]
    a = [l / (pb.weno_eps + bk) ** 2 for l, bk in zip((0.1, 0.6, 0.3), b)]
    return sum(ak * qk for ak, qk in zip(a, q)) / sum(a)


def _dissipation(pb, r, v, T, p, Rm, Gm, V, G, at):
    """-1/2 T^t R |Lambda| Y [[W]] at the interfaces; at(a, j): node j = 0..5 of the stencil."""
    N, d = pb.N, pb.d
    nc = pb.nc
    L = torch.sqrt(sum(g * g for g in G[1:]))
    n = [g / L for g in G[1:]]
    one, zero = torch.ones_like(L), torch.zeros_like(L)
    if d == 2:
        T3 = [[n[0], n[1]], [-n[1], n[0]]]
    else:
        h = torch.sqrt(n[0] * n[0] + n[1] * n[1])
        hs = torch.where(h > 0, h, one)
        ct, st = torch.where(h > 0, n[0] / hs, one), torch.where(h > 0, n[1] / hs, zero)
        T3 = [[n[0], n[1], n[2]], [-st, ct, zero], [-n[2] * ct, -n[2] * st, h]]
    mean = lambda a: 0.5 * (at(a, 2) + at(a, 3))  # noqa: E731
    lm = lambda a: _lm(at(a, 2), at(a, 3))  # noqa: E731
    vb = [mean(v[m]) for m in range(d)]
    vh = [sum(T3[m][j] * vb[j] for j in range(d)) for m in range(d)]
    v2 = sum(m * m for m in vh)
    Tb = 1.0 / lm(1.0 / T)
    lr = [lm(r[l]) for l in range(N)]
    if N == 1:
        Rb, Gb, rho, Y = pb.R(0) * one, pb.gamma[0] * one, lr[0], [one]
        H = pb.gamma[0] * pb.cv[0] * Tb + 0.5 * v2
    else:
        Rb, Gb, rho = mean(Rm), mean(Gm), lm(r[0] + r[1])
        Y = [q / rho for q in lr]
        H = (mean(p) + sum(pb.cv[l] * lr[l] * Tb + pb.pinf[l] for l in range(N))) / rho + 0.5 * v2
    c = torch.sqrt(Rb * Gb * Tb)
    lam = (G[0] + L * vh[0]).abs() + L * c
    cols = []
    pre = torch.sqrt(rho / (Gb * Rb))
    for s in (-1.0, 1.0):
        col = list(Y) + [vh[0] + s * c] + vh[1:] + [H + s * c * vh[0]]
        cols.append([pre / math.sqrt(2.0) * q for q in col])
    if N == 1:
        se = torch.sqrt(rho / (pb.cv[0] * pb.gamma[0]))
        cols.append([se] + [se * m for m in vh] + [se * 0.5 * v2])
    else:
        E = [0.5 * v2 - ((pb.cv[l] + pb.R(l)) * Tb - Gb * pb.cv[l] * Tb) / (Gb - 1) for l in range(2)]
        R1, R2 = pb.R(0), pb.R(1)
        sy, sg = torch.sqrt(Y[0] * Y[1]), torch.sqrt(Gb - 1)
        for da, db in ((-pre * sy * torch.sqrt(Gb * R2 / R1), pre * sy * torch.sqrt(Gb * R1 / R2)), (pre * Y[0] * sg, pre * Y[1] * sg)):
            cols.append([da, db] + [(da + db) * m for m in vh] + [da * E[0] + db * E[1]])
    for m in range(1, d):
        ss = torch.sqrt(rho * Tb) if N == 1 else pre * c
        cols.append([zero] * N + [ss if j == m else zero for j in range(d)] + [ss * vh[m]])
    nv = sum(torch.sqrt(sum(at(V[q], j) ** 2 for q in range(nc))) for j in (2, 3))
    weno = _weno_js if pb.weno else _weno_mr
    D = [zero] * nc
    for col in cols:
        rc = col[:N] + [sum(T3[m][j] * col[N + m] for m in range(d)) for j in range(d)] + [col[N + d]]
        w = [sum(rc[q] * at(V[q], j) for q in range(nc)) for j in range(6)]
        jw = weno(pb, (w[5], w[4], w[3], w[2], w[1])) - weno(pb, (w[0], w[1], w[2], w[3], w[4]))
        jp = w[3] - w[2]
        sig = jp.abs() > 1e-12 * torch.sqrt(sum(q * q for q in rc)) * nv
        cf = torch.where(sig & (torch.sign(jw) * torch.sign(jp) > 0), lam * jw, zero)
        D = [D[q] + rc[q] * cf for q in range(nc)]
    return -0.5 * torch.stack(D)


def _rhs64(pb, JU, J, x, xdot):
    dJU, dJ = torch.zeros_like(JU), torch.zeros_like(J)
    U = JU / J
    for k in range(pb.d):
        n = pb.n[k]
        Ue = _ext_U(pb, U, k, 3)
        rho, v, T, p, Rm, Gm = _prim(pb, Ue)
        r = [Ue[l] for l in range(pb.N)]
        row = _metrics_row(pb, x, k)
        xd = _ext_x(pb, xdot, k, 3, vel=True)
        M = [-sum(xd[j] * row[j] for j in range(pb.d))] + row
        beta = 1.0 / T
        cut = lambda a, s, m: _sl(a, k, s, m)  # noqa: E731
        f = 0.0
        for m in (1, 2, 3):
            w = n + 6 - m
            A = ([cut(q, 0, w) for q in r], [cut(q, 0, w) for q in v], cut(beta, 0, w), [cut(q, 0, w) for q in M])
            B = ([cut(q, m, w) for q in r], [cut(q, m, w) for q in v], cut(beta, m, w), [cut(q, m, w) for q in M])
            P = _pair(pb, A, B)
            f = f + _ALPHA[m - 1] * sum(cut(P, 2 - s, n + 1) for s in range(m))
        at = lambda a, j: _sl(a, k, j, n + 1)  # noqa: E731
        G = [sum(_ALPHA[m - 1] * 0.5 * sum(at(q, 2 - s) + at(q, 2 - s + m) for s in range(m)) for m in (1, 2, 3)) for q in M]
        if pb.es:
            f = f + _dissipation(pb, r, v, T, p, Rm, Gm, _entropy_vars(pb, Ue, v, T), G, at)
        dJU -= (cut(f, 1, n) - cut(f, 0, n)) / pb.dxi[k]
        dJ -= (cut(G[0], 1, n) - cut(G[0], 0, n)) / pb.dxi[k]
    return dJU, dJ


def _mesh64(pb, JU, J, x):
    U = JU / J
    rho, v, T, p, Rm, Gm = _prim(pb, U)
    c = torch.sqrt(Rm * Gm * T)
    s = 0.0
    for k in range(pb.d):
        row = [_sl(q, k, 3, pb.n[k]) for q in _metrics_row(pb, x, k)]
        s = s + (sum(q * m for q, m in zip(row, v)).abs() + c * torch.sqrt(sum(q * q for q in row))) / J / pb.dxi[k]
    dt = pb.cfl / s.max()
    one = torch.ones((), dtype=torch.float64, device=x.device)
    if pb.fixed_mesh:
        return torch.zeros_like(x), dt, one

    def sigma(kind, U):
        if kind == W.SIG_RHO1:
            return U[0]
        if kind == W.SIG_P:
            return _prim(pb, U)[3]
        return sum(U[l] for l in range(pb.N))

    th = torch.ones_like(J)
    for kind, al in zip(pb.sigma, pb.alpha):
        g2 = 0.0
        for k in range(pb.d):
            e = sigma(kind, _ext_U(pb, U, k, 1))
            g2 = g2 + ((_sl(e, k, 2, pb.n[k]) - _sl(e, k, 0, pb.n[k])) / (2 * pb.dxi[k])) ** 2
        g = torch.sqrt(g2)
        th = th + al * (g / g.max()) ** 2
    th = torch.sqrt(th)
    for _ in range(pb.nf):
        for k in range(pb.d):
            e, n = _ext_s(pb, th, k, 1), pb.n[k]
            th = 0.25 * (_sl(e, k, 0, n) + _sl(e, k, 2, n)) + 0.5 * _sl(e, k, 1, n)
    y = x
    wts = []
    for k in range(pb.d):
        e, n = _ext_s(pb, th, k, 1), pb.n[k]
        wts.append([0.5 * (th + _sl(e, k, o, n)) / pb.dxi[k] ** 2 for o in (0, 2)])
    den = sum(a + b for a, b in wts)
    for _ in range(pb.mu):
        num = 0.0
        for k in range(pb.d):
            e, n = _ext_x(pb, y, k, 1), pb.n[k]
            num = num + wts[k][0] * _sl(e, k, 0, n) + wts[k][1] * _sl(e, k, 2, n)
        y = num / den
    dtau = one
    for k in range(pb.d):
        e, n = _ext_x(pb, x, k, 1)[k], pb.n[k]
        dx = y[k] - x[k]
        up, dn = (_sl(e, k, 2, n) - x[k]) / (2 * dx), -(x[k] - _sl(e, k, 0, n)) / (2 * dx)
        b = torch.where(dx > 0, up, torch.where(dx < 0, dn, torch.ones_like(dx)))
        dtau = torch.minimum(dtau, b.min())
    return dtau * (y - x) / dt, dt, dtau


def _step64(pb, JU, J, x):
    xdot, dt, dtau = _mesh64(pb, JU, J, x)
    U1, J1, x1 = JU, J, x
    for a, b in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
        dU, dJ = _rhs64(pb, U1, J1, x1, xdot)
        U1, J1, x1 = a * JU + b * (U1 + dt * dU), a * J + b * (J1 + dt * dJ), a * x + b * (x1 + dt * xdot)
    return U1, J1, x1, xdot, torch.stack([dt, dtau])


def exact(case, seed):
    inst, _ = _initial(case, seed)
    if case["call"] == "batch":
        got = [_step64(pb, JU, J, x) for pb, JU, J, x, _ in inst]
        return {"state": torch.cat([a.reshape(-1) for g in got for a in g[:3]]),
                "xdot": torch.cat([g[3].reshape(-1) for g in got]), "dt": torch.stack([g[4] for g in got])}
    pb, JU, J, x, xdot = inst[0]
    if case["call"] == "diag":
        xdot = torch.zeros_like(x) if xdot is None else xdot
        dJU, dJ = _rhs64(pb, JU, J, x, xdot)
        U = JU / J
        rho, v, T, p, _, _ = _prim(pb, U)
        V = _entropy_vars(pb, U, v, T)
        eta = -sum(U[l] * (pb.cv[l] * torch.log(T) - pb.R(l) * torch.log(U[l])) for l in range(pb.N))
        phi = sum(pb.R(l) * U[l] - pb.pinf[l] / T for l in range(pb.N))
        vol = math.prod(pb.dxi[: pb.d])
        ent = torch.stack([vol * ((V * dJU).sum() - (phi * dJ).sum()), vol * (J * eta).sum()])
        g2 = 0.0
        rows = [[_sl(q, k, 3, pb.n[k]) for q in _metrics_row(pb, x, k)] for k in range(pb.d)]
        dr = []
        for k in range(pb.d):
            e = sum(_ext_U(pb, U, k, 1)[l] for l in range(pb.N))
            dr.append((_sl(e, k, 2, pb.n[k]) - _sl(e, k, 0, pb.n[k])) / (2 * pb.dxi[k]))
        for j in range(pb.d):
            g2 = g2 + (sum(rows[k][j] * dr[k] for k in range(pb.d)) / J) ** 2
        g = torch.sqrt(g2)
        psi = (30.0 * U[0] + (150.0 * U[1] if pb.N == 2 else 0.0)) / rho
        return {"dJU": dJU, "dJ": dJ, "entropy": ent, "phi": torch.exp(-psi * g / g.max())}
    JU, J, x, xdot, dt = _step64(pb, JU, J, x)
    if case["call"] == "host":
        return {"JU": JU, "J": J, "x": x, "t": dt[0]}
    return {"JU": JU, "J": J, "x": x, "xdot": xdot, "dt": dt}
