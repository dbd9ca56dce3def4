"""What a user of this framework has it compute, as cases that can be prepared, run and timed.

A case is a dict of plain numbers and texts.  `family` names the entry point's use:
  charges   pc_fields of point charges with sampled trajectories (the paper's Sec. 4.1, Listing 1)
  dipoles   pc_fields / pc_fields_plane of oscillating dipoles (the field grid of the benchmark)
  param     pc_fields_param of charges on analytic trajectories (Sec. 3.1's predefined charges)
  pairs     pc_dipoles_run of a batch of two-oscillator configurations (the separation sweep, Sec. 4.2)
  ring      pc_dipoles_run of oscillators on a ring
  cloud     pc_dipoles_run of oscillators in a cube
  moving    pc_dipoles_run_moving of a ring whose origins oscillate (Sec. 4.3)
  adjoint   pc_dipoles_adjoint of a ring (gradients of the final energy)
Physical parameters are those of the paper's listings and of this repository's workloads: charges of
one e and electron masses, 200 THz oscillators of 10 pm amplitude, steps of 1 as.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2107_12437_gb300 as pc

C = 299792458.0
E_CHARGE = 1.602176634e-19
M_E = 9.1093837015e-31
EPS0 = 8.8541878128e-12
KE = 1.0 / (4.0 * math.pi * EPS0)
DT = 1e-18
L = C * DT
OMEGA0 = 2 * math.pi * 200e12
SAMPLES = 15001        # history samples of the field sums' dipoles (15 fs)
ORBIT_SAMPLES = 10001  # of the orbiting charges (10 fs)


def listed():
    return [
        # the smallest call: the paper's Listing-1 use, two charges and a 101 x 101 grid of points in
        # one frame, in the default precision; launches and the call itself count
        dict(name="orbit_list_f64", family="charges", M=2, P=101 * 101, T=1, precision="f64", kind="total"),
        # fields of a set of dipoles at scattered detector points (a ragged list), mixed precision
        dict(name="dipoles_list_mixed", family="dipoles", shape="list", N=64, P=100003, T=2, precision="mixed",
             kind="total", amp=1e-11),
        # the benchmark's field grid: a movie of 16 frames on a 2048 x 2048 plane
        dict(name="grid_mixed", family="dipoles", shape="plane", N=64, nu=2048, nv=2048, T=16, precision="mixed",
             kind="total", amp=1e-11),
        # the same sources on an odd-sized plane in the all-float64 path
        dict(name="grid_f64", family="dipoles", shape="plane", N=64, nu=301, nv=517, T=1, precision="f64",
             kind="total", amp=1e-11),
        # predefined charges on their exact trajectories: an orbiting pair on a 1024 x 1024 grid
        dict(name="param_grid", family="param", M=2, P=1024 * 1024, T=1, kind="total"),
        # the separation sweep in full: 256 pairs from 1 nm to 1 um, 40 000 steps, mixed and float64
        dict(name="pairs_mixed", family="pairs", B=256, sep_lo=1e-9, sep_hi=1e-6, steps=40000, precision="mixed",
             orientation="s"),
        dict(name="pairs_f64", family="pairs", B=256, sep_lo=1e-9, sep_hi=1e-6, steps=10000, precision="f64",
             orientation="s"),
        # 256 oscillators on a 200 nm ring: many causal blocks of little work each, mixed and float64
        dict(name="ring_mixed", family="ring", N=256, steps=4000, precision="mixed"),
        dict(name="ring_f64", family="ring", N=256, steps=1000, precision="f64"),
        # 4096 oscillators in a 600 nm cube, the largest self-consistent run of this repository
        dict(name="cloud_mixed", family="cloud", N=4096, steps=1000, precision="mixed"),
        # the ring with oscillating origins
        dict(name="moving_ring_mixed", family="moving", N=256, steps=1000, precision="mixed"),
        # gradients of the ring's final energies (forward and reverse)
        dict(name="ring_adjoint", family="adjoint", N=256, steps=400, precision="f64"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    family = rng.choice(["charges", "dipoles", "dipoles", "dipoles", "param", "pairs", "ring", "cloud", "cloud",
                         "moving", "adjoint"])
    kind = rng.choice(["total", "total", "total", "coulomb", "radiation"])
    precision = rng.choice(["mixed", "mixed", "f64"])
    if family == "charges":
        M = rng.randint(1, 8)
        return dict(family=family, M=M, P=int(_log(rng, 300, 2e6 / M)), T=rng.randint(1, 5), precision=precision,
                    kind=kind)
    if family == "dipoles":
        N = int(_log(rng, 1, 300))
        T = rng.randint(1, 20)
        # a mixed case of up to 3e9, a float64 one of up to 1e8 (point, dipole, frame) triples
        most = (3e9 if precision == "mixed" else 1e8) / (N * T)
        P = int(_log(rng, 200, max(400, min(4e6, most))))
        c = dict(family=family, N=N, T=T, precision=precision, kind=kind, amp=_log(rng, 2e-12, 5e-11))
        if rng.random() < 0.4:
            return dict(c, shape="list", P=P)
        nu = max(1, min(P, int(math.sqrt(P) * _log(rng, 0.4, 2.5))))
        return dict(c, shape="plane", nu=nu, nv=max(1, P // nu))
    if family == "param":
        M = rng.randint(1, 6)
        return dict(family=family, M=M, P=int(_log(rng, 300, 4e6 / M)), T=rng.randint(1, 3), kind=kind)
    if family == "pairs":
        lo = _log(rng, 1e-9, 1e-7)
        return dict(family=family, B=int(_log(rng, 1, 300)), sep_lo=lo, sep_hi=lo * _log(rng, 2, 1e3),
                    steps=int(_log(rng, 200, 20000)), precision=precision, orientation=rng.choice(["s", "p"]))
    if family == "ring":
        N = int(_log(rng, 8, 400))
        return dict(family=family, N=N, steps=int(_log(rng, 100, 4000 if precision == "mixed" else 1000)),
                    precision=precision)
    if family == "cloud":
        N = int(_log(rng, 3, 5000 if precision == "mixed" else 1000))
        most = (1.5e10 if precision == "mixed" else 2e8) / (N * N)
        return dict(family=family, N=N, steps=int(_log(rng, 100, max(200, min(4000, most)))), precision=precision)
    if family == "moving":
        N = int(_log(rng, 8, 300))
        return dict(family=family, N=N, steps=int(_log(rng, 100, 1000 if precision == "mixed" else 300)),
                    precision=precision)
    N = int(_log(rng, 3, 300))
    return dict(family=family, N=N, steps=int(_log(rng, 100, 400)), precision=precision)


# ------------------------------------------------------------------------------------------------
# inputs, from the seed alone
# ------------------------------------------------------------------------------------------------
_KIND = {"total": pc.PC_TOTAL, "coulomb": pc.PC_COULOMB, "radiation": pc.PC_RADIATION}
_PREC = {"f64": pc.PC_F64, "mixed": pc.PC_MIXED}


def _unit(rng, n):
    v = rng.standard_normal((n, 3))
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _gpu(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64).cuda()


def _frames(T):
    # the last 5 fs of the dipoles' 15 fs, as the frames of a movie
    return [10e-15 + f * (5e-15 / T) for f in range(T)]


def _orbits(case, rng):
    """Charges +-e in turn on circles of about 1 nm within some nm of the origin, up to 0.1 c; the first rests."""
    M = case["M"]
    centre = np.zeros((M, 3))
    centre[2:] = rng.uniform(-5e-9, 5e-9, (max(0, M - 2), 3))
    e1 = _unit(rng, M)
    e2 = np.cross(e1, _unit(rng, M))
    e2 /= np.linalg.norm(e2, axis=1, keepdims=True)
    radius = rng.uniform(0.8e-9, 1.2e-9, M)
    w = rng.uniform(0.02, 0.1, M) * C / radius
    phase = rng.uniform(0, 2 * math.pi, M)
    if M > 1:
        radius[0] = 0.0
    q = E_CHARGE * np.where(np.arange(M) % 2 == 0, 1.0, -1.0)
    return centre, e1, e2, radius, w, phase, q


def _detectors(rng, P):
    """P points of a plane grid's extent (+-50 nm) a little off the charges' plane."""
    p = rng.uniform(-50e-9, 50e-9, (P, 3))
    p[:, 2] = rng.uniform(3e-9, 9e-9) * np.where(p[:, 2] > 0, 1.0, -1.0)
    return p


def _dipole_sources(case, rng):
    """Oscillating dipoles at random places of a 1 um cube, random axes: d(t) = e amp sin(omega0 t)."""
    N = case["N"]
    t = torch.arange(SAMPLES, dtype=torch.float64, device="cuda") * DT
    one = torch.ones((N, 1), dtype=torch.float64, device="cuda")
    s = E_CHARGE * case["amp"]
    d = dict(origin=_gpu(rng.uniform(0.0, 1e-6, (N, 3))), axis=_gpu(_unit(rng, N)), q=E_CHARGE * one[:, 0],
             m1=M_E * one[:, 0], m2=M_E * one[:, 0], d=one * (s * torch.sin(OMEGA0 * t)),
             d_dot=one * (s * OMEGA0 * torch.cos(OMEGA0 * t)),
             d_ddot=one * (-s * OMEGA0 * OMEGA0 * torch.sin(OMEGA0 * t)), t0=0.0, dt=DT)
    return SimpleNamespace(**d)


def _oscillators(case, rng):
    """(origin [B][N][3], axis, omega0 [B][N]) of the oscillator families."""
    f = case["family"]
    if f == "pairs":
        B = case["B"]
        sep = np.geomspace(case["sep_lo"], case["sep_hi"], B) * rng.uniform(1.0, 1.01)
        origin = np.zeros((B, 2, 3))
        origin[:, 1, 1 if case["orientation"] == "s" else 0] = sep
        axis = np.zeros((B, 2, 3))
        axis[:, :, 0] = 1.0
        return origin, axis, np.full((B, 2), OMEGA0)
    N = case["N"]
    if f == "cloud":
        # one oscillator in each of the first N cells of a lattice of 37.5 nm (the density of 4096 in
        # a 600 nm cube), anywhere in the cell but its last 5 nm: no two closer than that
        g = int(math.ceil(N ** (1 / 3) - 1e-9))
        cell = np.stack(np.unravel_index(rng.permutation(g ** 3)[:N], (g, g, g)), axis=1)
        origin = cell * 37.5e-9 + rng.uniform(0.0, 32.5e-9, (N, 3))
        return origin[None], _unit(rng, N)[None], np.full((1, N), OMEGA0)
    # rings: neighbours as far apart as 256 on a radius of 200 nm
    radius = 200e-9 * N / 256
    ang = 2 * math.pi * np.arange(N) / N + rng.uniform(0, 2 * math.pi)
    origin = np.stack([radius * np.cos(ang), radius * np.sin(ang), np.zeros(N)], axis=1)[None]
    axis = np.zeros((1, N, 3))
    axis[..., 2] = 1.0
    return origin, axis, OMEGA0 * (1.0 + rng.uniform(-0.01, 0.01, (1, N)))


def _inputs(case, seed):
    """Everything a pass needs, in numbers, without the framework."""
    rng = np.random.default_rng([int(seed), 2107])
    f = case["family"]
    if f == "charges":
        centre, e1, e2, radius, w, phase, q = _orbits(case, rng)
        t = np.arange(ORBIT_SAMPLES) * DT
        a = w[:, None] * t[None] + phase[:, None]
        c, s = np.cos(a)[..., None], np.sin(a)[..., None]
        r, ww = radius[:, None, None], w[:, None, None]
        u, v = e1[:, None], e2[:, None]
        src = SimpleNamespace(q=_gpu(q), pos=_gpu(centre[:, None] + r * (c * u + s * v)),
                              vel=_gpu(r * ww * (c * v - s * u)), acc=_gpu(-r * ww * ww * (c * u + s * v)), t0=0.0,
                              dt=DT, static_before=1)
        times = [10e-15 - 1e-16 * k for k in range(case["T"])]
        return SimpleNamespace(src=src, points=_gpu(_detectors(rng, case["P"])), times=times)
    if f == "param":
        centre, e1, e2, radius, w, phase, q = _orbits(case, rng)
        M = case["M"]
        par = np.zeros((M, 12))
        kind = np.full(M, pc.PC_TRAJ_CIRCULAR, dtype=np.int32)
        par[:, :3], par[:, 3:6], par[:, 6:9], par[:, 9], par[:, 10], par[:, 11] = centre, e1, e2, radius, w, phase
        if M > 1:
            kind[0] = pc.PC_TRAJ_STATIONARY
        times = [10e-15 + 1e-16 * k for k in range(case["T"])]
        return SimpleNamespace(kind=torch.as_tensor(kind).cuda(), q=_gpu(q), par=_gpu(par),
                               points=_gpu(_detectors(rng, case["P"])), times=times)
    if f == "dipoles":
        src = _dipole_sources(case, rng)
        times = _frames(case["T"])
        if case["shape"] == "list":
            return SimpleNamespace(src=src, points=_gpu(rng.uniform(0.0, 1e-6, (case["P"], 3))), times=times)
        z = rng.uniform(0.45e-6, 0.55e-6)
        du, dv = 1e-6 / max(1, case["nu"] - 1), 1e-6 / max(1, case["nv"] - 1)
        plane = dict(origin=(0.0, 0.0, z), eu=(du, 0.0, 0.0), ev=(0.0, dv, 0.0), nu=case["nu"], nv=case["nv"])
        return SimpleNamespace(src=src, plane=plane, times=times)
    origin, axis, omega0 = _oscillators(case, rng)
    one = np.ones(omega0.shape)
    dp = SimpleNamespace(origin=_gpu(origin), axis=_gpu(axis), q=_gpu(E_CHARGE * one), m1=_gpu(M_E * one),
                         m2=_gpu(M_E * one), omega0=_gpu(omega0), d0=_gpu(E_CHARGE * 1e-11 * one))
    s = SimpleNamespace(dp=dp, steps=case["steps"])
    if f == "moving":
        # origins oscillating along x by 1 A at 20 THz (half steps)
        om, amp = 2 * math.pi * 20e12, 1e-10 * rng.uniform(0.5, 1.0, omega0.shape)
        t = torch.arange(2 * s.steps + 1, dtype=torch.float64, device="cuda") * (DT / 2)
        u = _gpu([1.0, 0.0, 0.0])
        x = _gpu(amp)[..., None, None] * u
        co, si = torch.cos(om * t)[:, None], torch.sin(om * t)[:, None]
        s.motion = (dp.origin[:, :, None] + (co - 1.0) * x, -om * si * x, -om * om * co * x)
    if f == "adjoint":
        s.weight = _gpu(rng.uniform(0.5, 1.5, omega0.shape))
    return s


# ------------------------------------------------------------------------------------------------
# the passes
# ------------------------------------------------------------------------------------------------
_context = None


def prepare(case, seed):
    global _context
    if _context is None:  # one context for the whole program
        _context = pc.Context(0)
    s = _inputs(case, seed)
    s.case, s.ctx = dict(case), _context
    return s


def run(s):
    c, f = s.case, s.case["family"]
    if f == "charges":
        return pc.pc_fields(s.ctx, charges=s.src, points=s.points, times=s.times, kind=_KIND[c["kind"]],
                            precision=_PREC[c["precision"]])
    if f == "dipoles":
        opts = dict(dipoles=s.src, times=s.times, kind=_KIND[c["kind"]], precision=_PREC[c["precision"]])
        if c["shape"] == "list":
            return pc.pc_fields(s.ctx, points=s.points, **opts)
        return pc.pc_fields_plane(s.ctx, **s.plane, **opts)
    if f == "param":
        return pc.pc_fields_param(s.ctx, s.kind, s.q, s.par, s.points, s.times, field_kind=_KIND[c["kind"]])
    if f == "moving":
        return pc.pc_dipoles_run_moving(s.ctx, s.dp, s.motion, DT, s.steps, precision=_PREC[c["precision"]])
    if f == "adjoint":
        return pc.pc_dipoles_adjoint(s.ctx, s.dp, DT, s.steps, s.weight, precision=_PREC[c["precision"]])
    return pc.pc_dipoles_run(s.ctx, s.dp, DT, s.steps, precision=_PREC[c["precision"]])


def _points(case):
    return case["nu"] * case["nv"] if case.get("shape") == "plane" else case["P"]


def work(case):
    """Each input read once, each output written once; operations of the plain per-charge method: 146 for
    a charge's E, B, phi and A at a point, 125 for its part of one driving field (an add or multiply 1)."""
    f = case["family"]
    if f in ("charges", "dipoles", "param"):
        P, T = _points(case), case["T"]
        out = (3 + 3 + 3 + 1) * (4 if case.get("precision") == "mixed" else 8) + 1
        pts = 0 if case.get("shape") == "plane" else 24 * P
        charges = 2 * case["N"] if f == "dipoles" else case["M"]
        src = {"charges": charges * ORBIT_SAMPLES * 72, "dipoles": charges // 2 * SAMPLES * 24,
               "param": charges * 108}[f]
        return {"bytes": P * T * out + pts + src, "flops": 146.0 * P * T * charges}
    B, N = case.get("B", 1), case.get("N", 2)
    S = case["steps"] + 1
    # two driving fields a step from two charges of every other oscillator, about 60 operations of RK4
    flops = B * N * case["steps"] * (2.0 * 2 * 125 * (N - 1) + 60)
    if f == "adjoint":  # a reverse pass costs at least what the forward one does, once more
        return {"bytes": B * N * (80 + 40), "flops": 2 * flops}
    moving = B * N * (2 * S - 1) * 72 if f == "moving" else 0
    return {"bytes": B * N * (80 + S * 32) + moving, "flops": flops}


# ------------------------------------------------------------------------------------------------
# the same in plain torch, float64
# ------------------------------------------------------------------------------------------------
def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _field(q, a, v, acc, kind="total", only_E=False):
    """Lienard-Wiechert fields (Griffiths): a = r - r_s, v, acc lists of three tensors at the retarded time."""
    R = torch.sqrt(_dot(a, a))
    u = [C * a[i] / R - v[i] for i in range(3)]
    Ru = C * R - _dot(a, v)
    f = KE * q * R / Ru ** 3
    g = (C * C - _dot(v, v)) if kind != "radiation" else torch.zeros_like(R)
    aa = _dot(a, acc)
    E = [f * ((g + (aa if kind != "coulomb" else 0.0)) * u[i] - (acc[i] * Ru if kind != "coulomb" else 0.0))
         for i in range(3)]
    if only_E:
        return E
    B = [x / (R * C) for x in _cross(a, E)]
    phi = KE * q * C / Ru
    return E, B, phi, [phi * v[i] / C ** 2 for i in range(3)]


def _retarded(r, u, sample, last, k):
    """Segment and fraction of the retarded time on a piecewise-linear history whose sample k is sample(k):
    c^2 (u - k - th)^2 dt^2 = |r - p(k + th)|^2, from a first guess of k; the third value: before sample 0."""
    for _ in range(4):
        kk = k.clamp(0, last - 1)
        p0, p1 = sample(kk), sample(kk + 1)
        a = [r[i] - p0[i] for i in range(3)]
        D = [p1[i] - p0[i] for i in range(3)]
        Tm = u - kk
        A = L * L - _dot(D, D)
        Bq = _dot(a, D) - L * L * Tm
        Cq = (L * Tm) ** 2 - _dot(a, a)
        th = Cq / (-Bq + torch.sqrt((Bq * Bq - A * Cq).clamp(min=0)))
        k = kk + torch.floor(th).to(torch.int64)
    p0 = sample(torch.zeros_like(kk))
    a = [r[i] - p0[i] for i in range(3)]
    return kk, th, L * u <= torch.sqrt(_dot(a, a))


def _lerp(f, kk, th, rest):
    x0, x1 = f(kk), f(kk + 1)
    return [torch.where(rest, torch.zeros_like(th), x0[i] + th * (x1[i] - x0[i])) for i in range(len(x0))]


def _add_fields(out, lo, hi, f, case, r, u, sources):
    for q, sample, vel, acc, last, k in sources:
        kk, th, rest = _retarded(r, u, sample, last, k)
        first = sample(torch.zeros_like(kk))
        p = _lerp(sample, kk, th, torch.zeros_like(rest))
        p = [torch.where(rest, first[i] + 0 * th, p[i]) for i in range(3)]
        E, B, phi, A = _field(q, [r[i] - p[i] for i in range(3)], _lerp(vel, kk, th, rest),
                              _lerp(acc, kk, th, rest), case["kind"])
        for i in range(3):
            out["E"][f, lo:hi, i] += E[i]
            out["B"][f, lo:hi, i] += B[i]
            out["A"][f, lo:hi, i] += A[i]
        out["phi"][f, lo:hi] += phi


def _exact_fields(case, s):
    P, T = _points(case), case["T"]
    if case["family"] != "param" and P * T * (2 * case["N"] if "N" in case else case["M"]) > 4e9:
        return None  # the whole movie takes too long this way
    z = dict(dtype=torch.float64, device="cuda")
    out = dict(E=torch.zeros((T, P, 3), **z), B=torch.zeros((T, P, 3), **z), phi=torch.zeros((T, P), **z),
               A=torch.zeros((T, P, 3), **z), mask=None)
    step = 1 << 20
    for lo in range(0, P, step):
        hi = min(P, lo + step)
        if case.get("shape") == "plane":
            i = torch.arange(lo, hi, device="cuda")
            pl = s.plane
            iu, iv = (i // pl["nv"]).double(), (i % pl["nv"]).double()
            r = [pl["origin"][c] + iu * pl["eu"][c] + iv * pl["ev"][c] for c in range(3)]
        else:
            r = [s.points[lo:hi, c].contiguous() for c in range(3)]
        for f, t in enumerate(s.times):
            if case["family"] == "param":
                _add_param(out, lo, hi, f, case, r, t, s)
                continue
            u = torch.full_like(r[0], t / DT)
            if case["family"] == "charges":
                x = s.src
                cols = [[h[m, :, c].contiguous() for c in range(3)] for m in range(case["M"])
                        for h in (x.pos, x.vel, x.acc)]
                src = []
                for m in range(case["M"]):
                    p, v, a = cols[3 * m: 3 * m + 3]
                    d = torch.sqrt(sum((r[c] - p[c][-1]) ** 2 for c in range(3)))
                    src.append((float(x.q[m]), lambda k, h=p: [y[k] for y in h], lambda k, h=v: [y[k] for y in h],
                                lambda k, h=a: [y[k] for y in h], ORBIT_SAMPLES - 1,
                                torch.floor(u - d / L).to(torch.int64)))
                _add_fields(out, lo, hi, f, case, r, u, src)
                continue
            x = s.src
            for j in range(case["N"]):
                o, ax, q = x.origin[j].tolist(), x.axis[j].tolist(), float(x.q[j])
                d = torch.sqrt(sum((r[c] - o[c]) ** 2 for c in range(3)))
                k = torch.floor(u - d / L).to(torch.int64)
                src = []
                for sign in (0.5, -0.5):
                    w = sign / q
                    src.append((2 * sign * q, lambda n, w=w, j=j: [o[c] + w * ax[c] * x.d[j][n] for c in range(3)],
                                lambda n, w=w, j=j: [w * ax[c] * x.d_dot[j][n] for c in range(3)],
                                lambda n, w=w, j=j: [w * ax[c] * x.d_ddot[j][n] for c in range(3)], SAMPLES - 1, k))
                _add_fields(out, lo, hi, f, case, r, u, src)
    return out


def _add_param(out, lo, hi, f, case, r, t, s):
    for m in range(case["M"]):
        par, q = s.par[m].tolist(), float(s.q[m])
        still = int(s.kind[m]) == pc.PC_TRAJ_STATIONARY
        rad, w, ph = (0.0, 0.0, 0.0) if still else par[9:12]

        def state(tt):
            c, n = torch.cos(w * tt + ph), torch.sin(w * tt + ph)
            e = [c * par[3 + i] + n * par[6 + i] for i in range(3)]
            return ([par[i] + rad * e[i] for i in range(3)],
                    [rad * w * (c * par[6 + i] - n * par[3 + i]) for i in range(3)],
                    [-rad * w * w * e[i] for i in range(3)])

        x = torch.full_like(r[0], t)
        for _ in range(30):  # fixed point t' = t - |r - r(t')| / c, contracting by v/c < 0.1 a pass
            p, _v, _a = state(x)
            x = t - torch.sqrt(sum((r[i] - p[i]) ** 2 for i in range(3))) / C
        p, v, acc = state(x)
        E, B, phi, A = _field(q, [r[i] - p[i] for i in range(3)], v, acc, case["kind"])
        for i in range(3):
            out["E"][f, lo:hi, i] += E[i]
            out["B"][f, lo:hi, i] += B[i]
            out["A"][f, lo:hi, i] += A[i]
        out["phi"][f, lo:hi] += phi


def _exact_run(case, s):
    """Algorithm 1 with RK4: the stage fields of K steps at once (their retarded times precede the first), then
    the K steps; dipoles rest at d0 for t <= 0."""
    dp, n_steps = s.dp, case["steps"]
    B, N = dp.q.shape
    dist = (dp.origin[:, :, None] - dp.origin[:, None]).norm(dim=-1)
    off = torch.eye(N, dtype=torch.bool, device="cuda")
    moved = 2e-10 if case["family"] == "moving" else 0.0
    K = int(max(1, min(16, math.floor((float(dist[:, ~off].min()) - moved - 3e-11) / (1.01 * L)))))
    blocks = -(-n_steps // K)
    if blocks * (1.0 + B * N * N * 2 * K / 1.2e6) * 4e-3 > 18.0:
        return None  # too long this way
    S = n_steps + 1
    z = dict(dtype=torch.float64, device="cuda")
    d, dd, ddd = (torch.zeros((B, N, S), **z) for _ in range(3))
    d[..., 0] = dp.d0
    m = dp.m1 * dp.m2 / (dp.m1 + dp.m2)
    g0 = dp.q ** 2 * dp.omega0 ** 2 / (6 * math.pi * EPS0 * C ** 3 * m)
    qm, w2 = dp.q ** 2 / m, dp.omega0 ** 2
    if case["family"] == "moving":
        org = [x.contiguous() for x in s.motion]
    else:
        org = [dp.origin[:, :, None], None, None]
    bj = torch.arange(B, device="cuda")[:, None, None, None]
    jj = torch.arange(N, device="cuda")[None, None, :, None]

    def at(x, h):  # a source quantity [B][N][*] at samples h [B][i][j][stage]
        return x[bj, jj, h]

    def origin(c, which, k):
        x = org[which]
        if x is None:
            return 0.0
        return at(x[..., c], 2 * k if x.shape[2] > 1 else torch.zeros_like(k))

    def drive(n0, half):  # E_d [B][N][len(half)] at times n0 + half / 2 (samples 0 .. n0 known)
        u = (n0 + 0.5 * half)[None, None, None, :].expand(B, N, N, -1)
        if case["family"] == "moving":
            hr = 2 * n0 + half
            r = [org[0][:, :, hr, c][:, :, None, :].expand(B, N, N, -1) for c in range(3)]
            here = [org[0][:, None, :, 2 * n0, c][..., None] for c in range(3)]
        else:
            r = [dp.origin[:, :, None, None, c].expand(B, N, N, u.shape[-1]) for c in range(3)]
            here = [dp.origin[:, None, :, None, c] for c in range(3)]
        k = torch.floor(u - torch.sqrt(sum((r[c] - here[c]) ** 2 for c in range(3))) / L).to(torch.int64)
        pj = [dp.axis[:, None, :, None, c] for c in range(3)]
        E = 0.0
        for sign in (0.5, -0.5):
            w = (sign / dp.q)[:, None, :, None]

            def sample(kk):
                x = w * at(d, kk)
                return [origin(c, 0, kk) + x * pj[c] for c in range(3)]

            def vel(kk):
                x = w * at(dd, kk)
                return [origin(c, 1, kk) + x * pj[c] for c in range(3)]

            def acc(kk):
                x = w * at(ddd, kk)
                return [origin(c, 2, kk) + x * pj[c] for c in range(3)]

            kk, th, rest = _retarded(r, u, sample, max(n0, 1), k)
            if n0 == 0:
                rest = torch.ones_like(rest)
            first = sample(torch.zeros_like(kk))
            p = _lerp(sample, kk, th, torch.zeros_like(rest))
            p = [torch.where(rest, first[c], p[c]) for c in range(3)]
            f = _field(2 * sign * dp.q[:, None, :, None], [r[c] - p[c] for c in range(3)], _lerp(vel, kk, th, rest),
                       _lerp(acc, kk, th, rest), only_E=True)
            E = E + sum(f[c] * dp.axis[:, :, None, None, c] for c in range(3))
        return torch.where(off[None, :, :, None], torch.zeros_like(E), E).sum(dim=2)

    e1 = drive(0, torch.zeros(1, dtype=torch.int64, device="cuda"))[..., 0]
    for n0 in range(0, n_steps, K):
        kb = min(K, n_steps - n0)
        Es = drive(n0, torch.arange(1, 2 * kb + 1, device="cuda"))
        y0, y1 = d[..., n0], dd[..., n0]
        for k in range(kb):
            e2, e4 = Es[..., 2 * k], Es[..., 2 * k + 1]
            k1a, k1b = y1, -g0 * y1 - w2 * y0 + qm * e1
            ya, yb = y0 + 0.5 * DT * k1a, y1 + 0.5 * DT * k1b
            k2a, k2b = yb, -g0 * yb - w2 * ya + qm * e2
            ya, yb = y0 + 0.5 * DT * k2a, y1 + 0.5 * DT * k2b
            k3a, k3b = yb, -g0 * yb - w2 * ya + qm * e2
            ya, yb = y0 + DT * k3a, y1 + DT * k3b
            k4a, k4b = yb, -g0 * yb - w2 * ya + qm * e4
            y0 = y0 + DT / 6 * (k1a + 2 * k2a + 2 * k3a + k4a)
            y1 = y1 + DT / 6 * (k1b + 2 * k2b + 2 * k3b + k4b)
            n = n0 + k + 1
            d[..., n], dd[..., n], ddd[..., n] = y0, y1, qm * e4 - g0 * y1 - w2 * y0
            e1 = e4
    energy = (m / (2 * dp.q ** 2))[..., None] * (w2[..., None] * d * d + dd * dd)
    return dict(d=d, d_dot=dd, d_ddot=ddd, energy=energy)


def exact(case, seed):
    if case["family"] == "adjoint":
        return None  # differentiating the run above takes far more memory than the run
    s = _inputs(case, seed)
    if case["family"] in ("charges", "dipoles", "param"):
        return _exact_fields(case, s)
    return _exact_run(case, s)
