"""What a user of the radiation library has it do, as cases that can be timed and checked.

Every case goes through the public entry points of paper_1802_03972_gb300.rad.  A pass of most kinds is what a
simulation does between two readouts: zero the accumulators, hand over the time steps' particles, read the spectra.

Kinds:
  steps    rad.Context, mixed precision: accumulate() per time step, then spectrum().  `literal` also keeps the
           paper's literal sum; `host` takes the particles from pinned host memory and returns the spectra there.
  push     the same without beta_dot: push_step() per time step, push_flush(), spectrum().
  batch    rad.Batch: several jobs' steps per round, then each job's spectrum().
  static   accumulate_static() into accumulators that the program owns.
  fp64     a rad.Context of precision PREC_FP64 (the check of a mixed run on part of its bunch).
  readout  spectra of accumulators resumed from a checkpoint: 1-D shape, 3-D box shape, two species.

The mixed path sums in FP32, and its readout widens the result to float64: the spectra of the mixed kinds are kept
as a program keeps them, in float32.  Those of the FP64 context and of the readout stay float64.
"""
import math
import struct
from decimal import Decimal, getcontext

import numpy as np
import torch

from paper_1802_03972_gb300 import rad

C = 299792458.0
Q_E, M_E, EPS0 = 1.602176634e-19, 9.1093837015e-31, 8.8541878128e-12
K0 = Q_E**2 / (16.0 * math.pi**3 * EPS0 * C)
DT = 1e-16           # time step of the betatron bunches, s
WIDTH = 0.1e-6       # macro-particle width, m


def listed():
    return [
        # a small diagnostic in a test run: 64 electrons on helices, a linear frequency grid, a line of directions;
        # launches and latency are all there is
        {"name": "helix", "kind": "steps", "bunch": "helix", "n": 64, "n_omega": 128, "nx": 16, "ny": 1, "steps": 16},
        # one small job alone, with ragged sizes: fewer bins and particles than the GPU has lanes for
        {"name": "job_small", "kind": "steps", "bunch": "betatron", "n": 1777, "n_omega": 96, "nx": 5, "ny": 5, "steps": 8},
        # an ordinary job of a host program: odd sizes, particles from and spectra to pinned host memory
        {"name": "job_host", "kind": "steps", "bunch": "betatron", "n": 9973, "n_omega": 200, "nx": 9, "ny": 7, "steps": 4,
         "host": True},
        # the LWFA-shaped bunch on its 512 x 256 grid: the benchmark's time step
        {"name": "lwfa", "kind": "steps", "bunch": "betatron", "n": 100000, "n_omega": 512, "nx": 16, "ny": 16, "steps": 1},
        # in-situ scale: one call of 1e6 macro-particles on 1024 frequencies, TSC shape
        {"name": "insitu", "kind": "steps", "bunch": "betatron", "n": 1000000, "n_omega": 1024, "nx": 16, "ny": 16, "steps": 1},
        # a call that holds a whole domain: particles over 2 mm, far beyond one reference point's phase range
        {"name": "wide", "kind": "steps", "bunch": "wide", "n": 100000, "n_omega": 512, "nx": 8, "ny": 8, "steps": 1},
        # the paper's literal per-particle sum beside the split
        {"name": "literal", "kind": "steps", "bunch": "betatron", "n": 30011, "n_omega": 512, "nx": 8, "ny": 8, "steps": 2,
         "literal": True},
        # in-situ coupling to a pusher that has no accelerations
        {"name": "push", "kind": "push", "bunch": "betatron", "n": 50000, "n_omega": 256, "nx": 8, "ny": 8, "steps": 4},
        # a parameter scan: 16 small jobs of different sizes advanced together
        {"name": "batch", "kind": "batch", "jobs": 16, "n_lo": 1000, "n_hi": 10000, "omega_hi": 256, "side_hi": 8, "steps": 8},
        # a plug-in that may not allocate device memory
        {"name": "static", "kind": "static", "bunch": "betatron", "n": 20000, "n_omega": 128, "nx": 4, "ny": 4, "steps": 4},
        # a check of the mixed path: part of a bunch and of the directions in FP64
        {"name": "fp64", "kind": "fp64", "bunch": "betatron", "n": 4001, "n_omega": 512, "nx": 4, "ny": 4, "steps": 1},
        # the readouts of the benchmark's 131072 bins
        {"name": "readout", "kind": "readout", "n_omega": 512, "nx": 16, "ny": 16},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "push", "batch", "static", "fp64", "readout"])
    if kind == "batch":
        lo = _log_int(rng, 200, 2000)
        return {"kind": kind, "jobs": rng.randint(3, 18), "n_lo": lo, "n_hi": lo * rng.randint(2, 10),
                "omega_hi": rng.choice([64, 128, 256, 512]), "side_hi": rng.choice([4, 8]), "steps": rng.randint(2, 8)}
    nx, ny = rng.randint(1, 16), rng.randint(1, 16)
    if kind == "readout":
        return {"kind": kind, "n_omega": _log_int(rng, 48, 1024), "nx": nx + 2, "ny": ny + 2}
    n_omega = _log_int(rng, 48, 1024)
    if kind == "static":
        n_omega = _log_int(rng, 48, 512)
        nx, ny = min(nx, 8), min(ny, 8)
        return {"kind": kind, "bunch": "betatron", "n": _log_int(rng, 500, 65536), "n_omega": n_omega, "nx": nx, "ny": ny,
                "steps": rng.randint(1, 4)}
    if kind == "fp64":
        nx, ny = min(nx, 5), min(ny, 5)
        top = int(2e8 / (n_omega * nx * ny))
        return {"kind": kind, "bunch": "betatron", "n": _log_int(rng, 200, max(201, min(20000, top))), "n_omega": n_omega,
                "nx": nx, "ny": ny, "steps": 1}
    steps = rng.randint(1, 8) if kind == "steps" else rng.randint(2, 6)
    top = int(4e10 / (n_omega * nx * ny * steps))  # (the largest listed case: 2.6e11 updates)
    c = {"kind": kind, "bunch": "betatron", "n": _log_int(rng, 300, max(301, min(1000000, top))), "n_omega": n_omega,
         "nx": nx, "ny": ny, "steps": steps}
    if kind == "steps":
        which = rng.choice(["device", "device", "host", "literal", "wide", "helix"])
        if which in ("host", "literal"):
            c[which] = True
        elif which != "device":
            c["bunch"] = which
        if which == "helix":
            c["n"] = min(c["n"], 2000)
        elif which == "host":
            c["n"] = min(c["n"], 200000)
    return c


# ------------------------------------------------------------------ inputs
def _omega(case):
    n = case["n_omega"]
    if case.get("bunch") == "helix":
        return np.linspace(1e15, 1e18, n)
    return 1e14 * 1e6 ** (np.arange(n) / (n - 1))


def _dirs(nx, ny):
    if ny == 1:
        t = np.linspace(0.0, 0.02, nx)
        return np.stack([np.sin(t), np.zeros(nx), np.cos(t)], axis=1)
    ty, tx = (a.ravel() for a in np.meshgrid(np.linspace(-0.01, 0.01, ny), np.linspace(-0.01, 0.01, nx), indexing="ij"))
    return np.stack([np.sin(tx) * np.cos(ty), np.sin(ty), np.cos(tx) * np.cos(ty)], axis=1)


def _bunch(case, seed):
    """[(r, beta, beta_dot, w, t, dt)] of the case's steps: float64 on the GPU, [3][n] and [n]."""
    g = np.random.Generator(np.random.PCG64(seed))
    n, dev = case["n"], torch.device("cuda")
    put = lambda a: torch.from_numpy(a).to(dev)  # noqa: E731
    out = []
    if case["bunch"] == "helix":  # gamma = 50, radius 1 um, undulator strength 1; w = 1
        ph0, bp, rho = put(g.uniform(0.0, 2 * math.pi, n)), 1.0 / 50.0, 1e-6
        wh, bz = bp * C / rho, math.sqrt(1.0 - 1.0 / 2500.0 - bp * bp)
        one = torch.ones(n, dtype=torch.float64, device=dev)
        for s in range(case["steps"]):
            t = s * 1e-17
            c, q = torch.cos(ph0 + wh * t), torch.sin(ph0 + wh * t)
            out.append((torch.stack([rho * c, rho * q, one * (bz * C * t)]), torch.stack([-bp * q, bp * c, bz * one]),
                        torch.stack([-bp * wh * c, -bp * wh * q, 0 * one]), one.clone(), t, 1e-17))
        return out
    # betatron motion at n_e = 1e18 cm^-3: sigma_r = 2 um, gamma log-normal about 300, w uniform in 1e3..1e5; along z
    # sigma = 1 um, or 2 mm uniform for a whole domain
    z0 = g.uniform(-1e-3, 1e-3, n) if case["bunch"] == "wide" else g.normal(0.0, 1e-6, n)
    z0, x0, y0 = put(z0), put(g.normal(0.0, 2e-6, n)), put(g.normal(0.0, 2e-6, n))
    gamma = put(300.0 * np.exp(0.1 * g.normal(0.0, 1.0, n)))
    px, py = put(g.uniform(0.0, 2 * math.pi, n)), put(g.uniform(0.0, 2 * math.pi, n))
    w = put(g.uniform(1e3, 1e5, n))
    kb = math.sqrt(1e24 * Q_E**2 / (EPS0 * M_E)) / C / torch.sqrt(2 * gamma)
    for s in range(case["steps"]):
        t = s * DT
        cx, sx, cy, sy = (f(kb * (C * t) + p) for p in (px, py) for f in (torch.cos, torch.sin))
        bx, by = -x0 * kb * sx, -y0 * kb * sy
        bz = torch.sqrt(1.0 - 1.0 / gamma**2 - bx * bx - by * by)
        ax, ay = -x0 * kb * kb * C * cx, -y0 * kb * kb * C * cy
        r = torch.stack([x0 * cx, y0 * cy, z0 + C * t * (1.0 - 0.5 / gamma**2)])
        out.append((r, torch.stack([bx, by, bz]), torch.stack([ax, ay, -(bx * ax + by * ay) / bz]), w.clone(), t, DT))
    return out


def _shape(case):
    if case.get("bunch") == "helix":
        return rad.FF_POINT, 0.0
    return (rad.FF_TSC if case["n_omega"] > 512 else rad.FF_GAUSS), WIDTH


def _jobs(case):
    """The jobs of a batch: sizes over the mix's ranges, the same for every seed."""
    g = np.random.Generator(np.random.PCG64(4500 + case["jobs"]))
    out = []
    for _ in range(case["jobs"]):
        n = int(round(math.exp(g.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        side = int(2 ** g.integers(2, int(math.log2(case["side_hi"])) + 1))
        out.append({"bunch": "betatron", "n": n, "n_omega": int(2 ** g.integers(6, int(math.log2(case["omega_hi"])) + 1)),
                    "nx": side, "ny": side, "steps": case["steps"]})
    return out


_HEADER = struct.Struct("<IIiiiiiiQ")  # the state blob's header (include/rad.h, multirank.py)


def _checkpoint(case, seed, species):
    """A mixed context's state blob [16][n_bins]: sums of both signs over six decades, and their compensations."""
    g = np.random.Generator(np.random.PCG64([seed, species]))
    bins = case["n_omega"] * case["nx"] * case["ny"]
    v = (g.normal(0.0, 1.0, (8, bins)) * 10.0 ** g.uniform(1.0, 7.0, bins)).astype(np.float32)
    comp = (v * g.uniform(-3e-8, 3e-8, (8, bins))).astype(np.float32)
    a = np.concatenate([v, comp])
    return a, _HEADER.pack(0x52414453, 1, 0, case["n_omega"], case["nx"] * case["ny"], 16, 4, 0, a.nbytes) + a.tobytes()


def _out(shape, host=False):
    new = lambda: torch.empty(shape, dtype=torch.float64, pin_memory=True) if host else torch.empty(shape, dtype=torch.float64, device="cuda")  # noqa: E731,E501
    return new(), new(), new()


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind == "batch":
        jobs = _jobs(case)
        data = [_bunch(j, seed + 1000 * i) for i, j in enumerate(jobs)]
        # one buffer that the program's pusher writes each round; the jobs' arrays are parts of it
        s["rounds"] = [torch.cat([a.reshape(-1) for d in data for a in d[k][:4]]) for k in range(case["steps"])]
        s["live"] = torch.empty_like(s["rounds"][0])
        at, parts = 0, []
        for j in jobs:
            n = j["n"]
            cut = [s["live"][at + 3 * n * i:at + 3 * n * (i + 1)] for i in range(3)] + [s["live"][at + 9 * n:at + 10 * n]]
            at += 10 * n
            parts.append((n, cut))
        s["steps"] = [[rad.make_step(n, *cut, d[k][4], d[k][5]) for (n, cut), d in zip(parts, data)]
                      for k in range(case["steps"])]
        s["ctx"] = [rad.Context(_omega(j), _dirs(j["nx"], j["ny"]), *_shape(j)) for j in jobs]
        s["batch"] = rad.Batch(s["ctx"])
        s["out"] = [_out((j["nx"] * j["ny"], j["n_omega"])) for j in jobs]
        return s
    omega, dirs = _omega(case), _dirs(case["nx"], case["ny"])
    shape = (len(dirs), len(omega))
    if kind == "readout":
        s["ctx"] = [rad.Context(omega, dirs, rad.FF_GAUSS, WIDTH) for _ in range(2)]
        for i, c in enumerate(s["ctx"]):
            c.state_import(_checkpoint(case, seed, i)[1])
        s["out"] = [_out(shape) for _ in range(3)]
        return s
    s["data"] = _bunch(case, seed)
    if kind == "static":
        s["omega"], s["dirs"] = torch.from_numpy(omega).cuda(), torch.from_numpy(dirs).cuda()
        s["state"] = torch.zeros((16, len(omega) * len(dirs)), dtype=torch.float32, device="cuda")
        return s
    s["ctx"] = rad.Context(omega, dirs, *_shape(case), prec=rad.PREC_FP64 if kind == "fp64" else rad.PREC_MIXED,
                           ff_flags=rad.FF_LITERAL if case.get("literal") else 0)
    host = bool(case.get("host"))
    if host:
        s["data"] = [tuple(a.cpu().pin_memory() for a in d[:4]) + d[4:] for d in s["data"]]
    s["out"] = _out(shape, host)
    s["lit"] = _out(shape)[0] if case.get("literal") else None
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "batch":
        for c in s["ctx"]:
            c.reset()
        for flat, steps in zip(s["rounds"], s["steps"]):
            s["live"].copy_(flat)
            s["batch"].accumulate(steps)
        return [[x.float() for x in c.spectrum(out=o)] for c, o in zip(s["ctx"], s["out"])]
    if kind == "readout":
        a, b = s["ctx"]
        return [a.spectrum(out=s["out"][0]), a.spectrum((rad.FF_CIC, WIDTH, rad.FF_3D), out=s["out"][1]),
                rad.spectrum_species([a, b], [(rad.FF_GAUSS, WIDTH), (rad.FF_TSC, 2 * WIDTH)], out=s["out"][2])]
    if kind == "static":
        s["state"].zero_()
        for d in s["data"]:
            rad.accumulate_static(s["omega"], s["dirs"], *d, s["state"])
        return s["state"][:8] - s["state"][8:]  # the accumulators' values: sums less their compensations
    ctx = s["ctx"]
    ctx.reset()
    if kind == "push":
        for r, beta, _, w, t, dt in s["data"]:
            ctx.push_step(r, beta, w, t, dt)
        ctx.push_flush()
    else:
        for d in s["data"]:
            ctx.accumulate(*d)
    out = ctx.spectrum(out=s["out"])
    if kind == "fp64":
        return list(out)
    out = [x.float() for x in out]
    if s["lit"] is not None:
        out.append(ctx.spectrum_literal(out=s["lit"]).float())
    return out


def work(case):
    """Per (particle, direction, frequency) of a step: the phase (4), sine and cosine (2), four complex multiply-adds
    with real weights (16).  Bytes: the particles (80, or 56 without beta_dot) and three float64 spectra per bin."""
    if case["kind"] == "batch":
        jobs = _jobs(case)
        up = sum(j["n"] * j["n_omega"] * j["nx"] * j["ny"] for j in jobs) * case["steps"]
        return {"bytes": sum(80 * j["n"] * case["steps"] + 24 * j["n_omega"] * j["nx"] * j["ny"] for j in jobs), "flops": 22 * up}
    bins = case["n_omega"] * case["nx"] * case["ny"]
    if case["kind"] == "readout":  # three readouts, the last of two species
        return {"bytes": bins * (64 * 4 + 24 * 3), "flops": bins * (4 * 24 + 3 * 20)}
    up = case["n"] * bins * case["steps"]
    per = 56 if case["kind"] == "push" else 80
    outs = 64 if case["kind"] == "static" else 32 if case.get("literal") else 24
    return {"bytes": per * case["n"] * case["steps"] + outs * bins, "flops": (34 if case.get("literal") else 22) * up}


# ------------------------------------------------------ the same in 64 bits
def _split(a):
    t = a * 134217729.0
    h = t - (t - a)
    return h, a - h


def _two_prod(a, b):
    p = a * b
    (ah, al), (bh, bl) = _split(a), _split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _two_sum(a, b):
    s = a + b
    v = s - a
    return s, (a - (s - v)) + (b - v)


def _inv_2pi():
    getcontext().prec = 50
    pi = Decimal("3.14159265358979323846264338327950288419716939937510582097494459")
    v = 1 / (2 * pi)
    return float(v), float(v - Decimal(float(v)))


def _turns(omega):
    """omega / 2 pi as a pair of doubles whose sum holds about 32 digits."""
    hi, lo = _inv_2pi()
    om = torch.from_numpy(omega).cuda()
    p, e = _two_prod(om, torch.full_like(om, hi))
    return p, e + om * lo


def _tau(n, r, t):
    """t - n.r/c as a pair of doubles."""
    hi, lo = torch.zeros_like(r[0]), torch.zeros_like(r[0])
    for i in range(3):
        p, e = _two_prod(r[i], torch.full_like(r[i], float(n[i])))
        hi, e2 = _two_sum(hi, p)
        lo = lo + e + e2
    q = hi / C
    p, e = _two_prod(q, torch.full_like(q, C))
    q_lo = ((hi - p) - e + lo) / C
    s, e = _two_sum(t, -q)
    return s, e - q_lo


def _form(kind, width, x):
    if kind == rad.FF_GAUSS:
        return np.exp(-0.5 * (x * width / C) ** 2)
    h = x * width / (2 * C)
    s = np.where(h == 0.0, 1.0, np.sin(h) / np.where(h == 0.0, 1.0, h))
    return {rad.FF_POINT: np.ones_like(x), rad.FF_CIC: s, rad.FF_TSC: s * s, rad.FF_QSC: s**3}[kind]


def _unit(dirs):
    return dirs / np.sqrt(dirs[:, :1] ** 2 + dirs[:, 1:2] ** 2 + dirs[:, 2:] ** 2)


def _sums(omega, dirs, data, f2=None):
    """Per direction: sums of a e^{i omega (t - n.r/c)} over all particles of all steps, [n_omega][3] complex, with
    weights w dt, sqrt(w) dt and, with f2, sqrt(w) sqrt(1 + (w - 1) f2) dt."""
    r, b, a = (torch.cat([d[i].reshape(3, -1) for d in data], dim=1) for i in range(3))
    w = torch.cat([d[3] for d in data])
    t = torch.cat([torch.full_like(d[3], d[4]) for d in data])
    dt = torch.cat([torch.full_like(d[3], d[5]) for d in data])
    fh, fl = _turns(omega)
    gh, gl = _split(fh)
    fh, fl, gh, gl = (v[:, None] for v in (fh, fl, gh, gl))
    f2 = None if f2 is None else torch.from_numpy(f2).cuda()[:, None]
    step = max(256, int(6e6 / len(omega)))
    for n in _unit(dirs):
        nv = torch.from_numpy(n).cuda()[:, None].expand_as(b)
        x = torch.linalg.cross(nv, torch.linalg.cross(nv - b, a, dim=0), dim=0)
        amp = (x / (1.0 - (nv * b).sum(0)) ** 2 * dt).T
        tau, tau_lo = _tau(n, r, t)
        ws = torch.cat([amp * w[:, None], amp * torch.sqrt(w)[:, None]], dim=1)
        total = torch.zeros((len(omega), 6 if f2 is None else 9), dtype=torch.complex128, device="cuda")
        for k in range(0, len(w), step):
            q, ql = tau[None, k:k + step], tau_lo[None, k:k + step]
            qh, qe = _split(q)
            p = fh * q
            e = ((gh * qh - p) + gh * qe + gl * qh) + gl * qe
            ph = ((p - torch.round(p)) + (e + (fh * ql + fl * q))) * (2 * math.pi)
            c, s = torch.cos(ph), torch.sin(ph)
            total[:, :6] += torch.complex(c @ ws[k:k + step], s @ ws[k:k + step])
            if f2 is not None:
                g = torch.sqrt(1.0 + (w[None, k:k + step] - 1.0) * f2)
                total[:, 6:] += torch.complex((c * g) @ ws[k:k + step, 3:], (s * g) @ ws[k:k + step, 3:])
        yield total


def _spectra(case, data):
    omega, dirs = _omega(case), _dirs(case["nx"], case["ny"])
    f2 = _form(*_shape(case), omega) ** 2
    rows = []
    for z in _sums(omega, dirs, data, f2 if case.get("literal") else None):
        z2 = (z.real**2 + z.imag**2).cpu().numpy()
        coh, inc = K0 * f2 * z2[:, :3].sum(1), K0 * (1 - f2) * z2[:, 3:6].sum(1)
        rows.append([coh, inc, coh + inc] + ([K0 * z2[:, 6:].sum(1)] if case.get("literal") else []))
    return [np.stack(v) for v in zip(*rows)]


def _push_data(data):
    out = []
    for i, d in enumerate(data):
        lo, hi = data[max(0, i - 1)], data[min(len(data) - 1, i + 1)]
        out.append((d[0], d[1], (hi[1] - lo[1]) / (hi[4] - lo[4]), d[3], d[4], d[5]))
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "readout":
        omega, n = _omega(case), _unit(_dirs(case["nx"], case["ny"]))
        u2, v2, u = [], [], []
        for i in range(2):
            a = _checkpoint(case, seed, i)[0].astype(np.float64)
            v = (a[:8] - a[8:]).reshape(8, len(n), len(omega))
            u.append(v[:4])
            u2.append((v[:4] ** 2).sum(0))
            v2.append((v[4:] ** 2).sum(0))
        out = []
        f1 = _form(rad.FF_GAUSS, WIDTH, omega)
        f3 = np.stack([np.prod([_form(rad.FF_CIC, WIDTH, omega * c) for c in d], axis=0) for d in n])
        for f in (f1, f3):
            coh, inc = K0 * f * f * u2[0], K0 * (1 - f * f) * v2[0]
            out.append([coh, inc, coh + inc])
        g = _form(rad.FF_TSC, 2 * WIDTH, omega)
        coh = K0 * ((f1 * u[0] + g * u[1]) ** 2).sum(0)
        inc = K0 * ((1 - f1 * f1) * v2[0] + (1 - g * g) * v2[1])
        return out + [[coh, inc, coh + inc]]
    if kind == "batch":
        if work(case)["flops"] > 2e11:
            return None
        return [_spectra(j, _bunch(j, seed + 1000 * i)) for i, j in enumerate(_jobs(case))]
    if work(case)["flops"] > 4e11:  # (over about 20 seconds)
        return None
    data = _bunch(case, seed)
    if kind == "push":
        data = _push_data(data)
    if kind != "static":
        return _spectra(case, data)
    # static: U and V along each direction's transverse basis (e1 from the axis least along n, e2 = n x e1)
    omega, dirs = _omega(case), _dirs(case["nx"], case["ny"])
    rows = []
    for n, z in zip(_unit(dirs), _sums(omega, dirs, data)):
        ax = 0
        ax = 1 if abs(n[1]) < abs(n[ax]) else ax
        ax = 2 if abs(n[2]) < abs(n[ax]) else ax
        e1 = np.eye(3)[ax] - n[ax] * n
        e1 /= np.sqrt((e1**2).sum())
        e = torch.from_numpy(np.stack([e1, np.cross(n, e1)], axis=1)).to(torch.complex128).cuda()
        uv = torch.cat([z[:, :3] @ e, z[:, 3:] @ e], dim=1)  # U.e1, U.e2, V.e1, V.e2
        rows.append(torch.stack([uv.real, uv.imag], dim=2).reshape(len(omega), 8).T)
    return torch.stack(rows, dim=1).reshape(8, -1)
