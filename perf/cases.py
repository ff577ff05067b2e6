"""What this framework is measured on: the work its users give it, through the public binding.

Kinds of work
  solve      the converged field solve delta -> phi, forces from a cold start (dgp_reset, dgp_solve_forces)
  steps      a segment of a PM run from a checkpoint: copy the state, dgp_reset, a few pm_step calls
  batch      the same segment for many small realisations at once (dgp_batch_step)
  adjoint    the backward of one step (pm_step_adjoint), the unit of a gradient through a run
  zeldovich  initial conditions from a linear field and their transpose
  snapshot   a snapshot in arbitrary particle order: cell sort, CIC deposit, P(k)
  bispectrum B and Q over a range of angles

Inputs are drawn on the GPU from the seed: power-law Gaussian fields (n_s = -1.5), Zel'dovich
particles of them, lognormal density contrasts (delta >= -1, skewed like an evolved field) and
particles sampled from such a contrast, in cell order as a run that sorts keeps them.
`exact` restates the method in 64 bits on torch.fft.  Positions come back unwrapped (continued
from where they started), since a coordinate within rounding of the box face may land on either
side of it.
"""
import math

import numpy as np
import torch

from paper_0906_4548_gb300 import dgp

OM = 0.27          # Omega_m0 of every workload in the repository
CH = 2997.92458    # c / H0, Mpc/h
W = 1.0 / 3.0      # splitting parameter
PRECISION = {"fp32": dgp.DGP_FP32, "mixed": dgp.DGP_MIXED, "fp64": dgp.DGP_FP64, "eft": dgp.DGP_MIXED_EFT,
             "f32r": dgp.DGP_MIXED_F32R}


def listed():
    return [
        # one 32^3 solve in double precision to 1e-10: a code check, the smallest call (launches and latency)
        {"name": "solve32_fp64", "kind": "solve", "n": 32, "box": 100.0, "a": 0.1, "rc": 1.0, "prec": "fp64",
         "rms": 1.0, "side": False},
        # one 64^3 solve at the binding's default precision on the default stream, as a notebook calls it
        {"name": "solve64_mixed", "kind": "solve", "n": 64, "box": 200.0, "a": 0.5, "rc": 1.0, "prec": "mixed",
         "rms": 1.6, "side": False},
        # one 128^3 solve at a = 1, the medium size of the solve and estimator workloads
        {"name": "solve128_fp32", "kind": "solve", "n": 128, "box": 200.0, "a": 1.0, "rc": 1.0, "prec": "fp32",
         "rms": 2.0, "side": True},
        # the largest mesh: one 512^3 solve
        {"name": "solve512_f32r", "kind": "solve", "n": 512, "box": 512.0, "a": 0.5, "rc": 1.0, "prec": "f32r",
         "rms": 1.6, "side": True},
        # a run on a mesh that is not a power of two, with the pair arithmetic for the residual
        {"name": "steps96_eft", "kind": "steps", "n": 96, "box": 150.0, "a": 0.3, "rc": 0.9, "prec": "eft",
         "rms": 1.9, "steps": 4, "side": True},
        # the flagship: 256^3 particles on a 256^3 mesh, box 400 Mpc/h, steps of a 200-step run
        {"name": "steps256_f32r", "kind": "steps", "n": 256, "box": 400.0, "a": 0.4, "rc": 1.0, "prec": "f32r",
         "rms": 2.0, "steps": 4, "side": True},
        # an ensemble of one small size: 16 realisations of 48^3 with different boxes and r_c
        {"name": "batch48", "kind": "batch", "n48": 16, "n64": 0, "n96": 0, "a": 0.3, "prec": "fp32", "rms": 1.8,
         "steps": 2},
        # a parameter scan over three sizes, unequal numbers of each
        {"name": "batch_ragged", "kind": "batch", "n48": 9, "n64": 7, "n96": 5, "a": 0.4, "prec": "fp32", "rms": 1.8,
         "steps": 2},
        # gradient of a 128^3 run: the transpose of one step (three field solves, two adjoint solves)
        {"name": "adjoint128_fp32", "kind": "adjoint", "n": 128, "box": 200.0, "a": 0.4, "rc": 1.0, "prec": "fp32",
         "rms": 1.5},
        # 256^3 initial conditions from a linear field, and the gradient's last stage back to it
        {"name": "zeldovich256", "kind": "zeldovich", "n": 256, "box": 400.0, "a": 0.02, "prec": "fp32", "rms": 0.5},
        # a snapshot read in arbitrary order (an odd number of particles): sort, deposit, P(k)
        {"name": "snapshot256", "kind": "snapshot", "n": 256, "box": 400.0, "np": 10000019, "prec": "fp32",
         "rms": 1.0},
        # bispectrum of a 128^3 field at eight angles
        {"name": "bispectrum128", "kind": "bispectrum", "n": 128, "box": 200.0, "k1": 0.5, "k2": 1.0, "nth": 8,
         "prec": "fp32", "rms": 1.0},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "steps", "steps", "batch", "adjoint", "zeldovich", "snapshot", "bispectrum"])
    a = round(_log_uniform(rng, 0.05, 1.0), 4)
    rms = round(rng.uniform(0.4, 2.0), 3)
    rc = round(rng.uniform(0.5, 2.0), 3)
    if kind == "batch":
        k = [rng.randint(1, 16), rng.randint(0, 16), rng.randint(0, 9)]
        return {"kind": kind, "n48": k[0], "n64": k[1], "n96": k[2], "a": round(rng.uniform(0.05, 0.5), 4),
                "prec": rng.choice(["fp32", "f32r", "eft"]), "rms": rms, "steps": rng.randint(1, 3)}
    prec = rng.choice(["fp32", "f32r", "f32r", "eft", "mixed", "fp64"])
    n = rng.choice({"solve": [16, 32, 48, 64, 96, 128, 256], "steps": [16, 32, 48, 64, 96, 128, 256],
                    "adjoint": [16, 32, 48, 64, 96, 128], "zeldovich": [32, 64, 128, 256],
                    "snapshot": [32, 64, 96, 128, 256], "bispectrum": [32, 64, 96, 128]}[kind])
    if n >= 128 and prec in ("mixed", "fp64"):
        prec = "f32r"
    if kind in ("zeldovich", "snapshot", "bispectrum"):
        prec = rng.choice(["fp32", "fp64"]) if n < 128 else "fp32"
    box = round(n * _log_uniform(rng, 1.2, 3.0), 2)
    c = {"kind": kind, "n": n, "box": box, "prec": prec, "rms": rms}
    if kind in ("solve", "steps", "adjoint", "zeldovich"):
        c["a"] = a if kind != "steps" else round(rng.uniform(0.05, 0.6), 4)
    if kind in ("solve", "steps", "adjoint"):
        c["rc"] = rc
    if kind in ("solve", "steps"):
        c["side"] = rng.random() < 0.7
    if kind == "steps":
        c["steps"] = rng.randint(1, 4)
    if kind == "snapshot":
        c["np"] = int(n ** 3 * rng.uniform(0.3, 1.0)) | 1
    if kind == "bispectrum":
        kf = 2.0 * math.pi / box
        c["k1"], c["k2"] = round(rng.uniform(3, n / 8) * kf, 4), round(rng.uniform(4, n / 8) * kf, 4)
        c["nth"] = rng.randint(1, 12)
    return c


# ---------------------------------------------------------------------------- inputs
def _axes(n, box):
    """k_x, k_y, k_z of the half grid (kz >= 0), broadcastable, and the Nyquist masks per axis."""
    i = torch.arange(n, device="cuda")
    s = torch.where(i < n // 2, i, i - n).double() * (2.0 * math.pi / box)
    z = torch.arange(n // 2 + 1, device="cuda").double() * (2.0 * math.pi / box)
    z[-1] = -z[-1]
    k = [s[:, None, None], s[None, :, None], z[None, None, :]]
    q = [(i == n // 2)[:, None, None], (i == n // 2)[None, :, None],
         (torch.arange(n // 2 + 1, device="cuda") == n // 2)[None, None, :]]
    return k, q


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _gauss_k(n, box, g, ns=-1.5):
    """Half spectrum of a Gaussian field with P ~ k^ns, unit variance on the mesh (float32 is ample for an input)."""
    k, q = _axes(n, box)
    k = [v.float() for v in k]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    amp = k2 ** (ns / 4.0)
    amp[0, 0, 0] = 0.0
    amp = amp.masked_fill(q[0] | q[1] | q[2], 0.0)
    f = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device="cuda")) * amp
    std = torch.fft.irfftn(f, s=(n, n, n)).std()
    return f / std


def _lognormal(n, box, rms, g, dtype):
    f = torch.fft.irfftn(_gauss_k(n, box, g), s=(n, n, n)) * rms
    f = torch.exp(f - 0.5 * rms * rms)
    return (f.double() / f.double().mean() - 1.0).to(dtype)


def _velocity_factor(a, rc):
    """a^2 E f with f = Omega_m(a)^0.68, a usual fit of the DGP growth rate."""
    E = _hubble(a, rc)
    return a * a * E * (OM * a ** -3 / (E * E)) ** 0.68


def _zeldovich(n, box, rms, g, vf, dtype):
    """Lattice particles displaced by Psi = i k / k^2 delta: (x, p), each (3, n^3)."""
    dk = _gauss_k(n, box, g) * rms
    k, q = _axes(n, box)
    k = [v.float() for v in k]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    x = torch.empty((3, n ** 3), dtype=dtype, device="cuda")
    p = torch.empty_like(x)
    lat = torch.arange(n, device="cuda").double() * (box / n)
    for j in range(3):
        psi = torch.fft.irfftn(1j * k[j] / k2 * dk, s=(n, n, n)).double()
        shape = [1, 1, 1]
        shape[j] = n
        xj = torch.remainder(lat.reshape(shape) + psi, box).to(dtype).reshape(-1)
        x[j] = torch.where(xj >= box, torch.zeros_like(xj), xj)
        p[j] = (vf * psi).reshape(-1).to(dtype)
    return x, p


def _evolved(n, box, rms, g, vf, dtype):
    """n^3 particles of a lognormal density, in cell order, moving with the linear flow of its Gaussian field."""
    m = n ** 3
    dk = _gauss_k(n, box, g) * rms
    f = torch.fft.irfftn(dk, s=(n, n, n)).double().reshape(-1)
    c = torch.cumsum(torch.exp(f - f.max()), 0)
    u = (torch.arange(m, device="cuda") + torch.rand(m, generator=g, device="cuda", dtype=torch.float64)) / m
    cell = torch.searchsorted(c, u * c[-1]).clamp_max(m - 1)
    del f, c, u
    k, _ = _axes(n, box)
    k = [v.float() for v in k]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = 1.0
    x = torch.empty((3, m), dtype=dtype, device="cuda")
    p = torch.empty_like(x)
    idx = [cell // (n * n), (cell // n) % n, cell % n]
    for j in range(3):
        psi = torch.fft.irfftn(1j * k[j] / k2 * dk, s=(n, n, n)).reshape(-1)[cell].double()
        off = torch.rand(m, generator=g, device="cuda", dtype=torch.float64)
        xj = ((idx[j] + off) * (box / n)).to(dtype)
        x[j] = torch.where(xj >= box, torch.zeros_like(xj), xj)
        p[j] = (vf * psi).to(dtype)
    return x, p


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _tol(case):
    return 1e-10 if case["prec"] == "fp64" else 1e-6


def _schedule(case):
    """Steps of a 200-step run from a = 0.02 to 1: uniform in ln a."""
    d = math.log(1.0 / 0.02) / 200
    return [case["a"] * math.exp(i * d) for i in range(case.get("steps", 1) + 1)]


def _members(case):
    """(mesh, box, r_c) of each realisation of a batch."""
    out = []
    for n in (48, 64, 96):
        for i in range(case["n%d" % n]):
            out.append((n, n * (1.1 + 0.11 * ((5 * i) % 16)), 0.5 + 0.1 * ((7 * i) % 16)))
    return out


def _inputs(case, seed):
    """The inputs alone, the same for the framework and for exact()."""
    g, t = _gen(seed), _dtype(case)
    kind = case["kind"]
    if kind == "solve":
        return {"delta": _lognormal(case["n"], case["box"], case["rms"], g, t)}
    if kind == "steps":
        x, p = _evolved(case["n"], case["box"], case["rms"], g, _velocity_factor(case["a"], case["rc"]), t)
        return {"x": x, "p": p}
    if kind == "batch":
        parts = [_evolved(n, box, case["rms"], g, _velocity_factor(case["a"], rc), t)
                 for n, box, rc in _members(case)]
        return {"x": [v[0] for v in parts], "p": [v[1] for v in parts]}
    if kind == "adjoint":
        x, p = _zeldovich(case["n"], case["box"], case["rms"], g, _velocity_factor(case["a"], case["rc"]), t)
        xb = torch.randn(x.shape, generator=g, device="cuda", dtype=t)
        pb = torch.randn(x.shape, generator=g, device="cuda", dtype=t)
        return {"x": x, "p": p, "xb": xb, "pb": pb}
    if kind == "zeldovich":
        n = case["n"]
        d = torch.fft.irfftn(_gauss_k(n, case["box"], g) * case["rms"], s=(n, n, n)).to(t)
        xb = torch.randn((3, n ** 3), generator=g, device="cuda", dtype=t)
        pb = torch.randn((3, n ** 3), generator=g, device="cuda", dtype=t)
        return {"delta": d, "xb": xb, "pb": pb}
    if kind == "snapshot":
        x, p = _zeldovich(case["n"], case["box"], case["rms"], g, 1.0, t)
        keep = torch.randperm(x.shape[1], generator=g, device="cuda")[:case["np"]]
        return {"x": x[:, keep].contiguous(), "p": p[:, keep].contiguous()}
    return {"delta": _lognormal(case["n"], case["box"], case["rms"], g, t)}


# ---------------------------------------------------------------------------- the framework
class State:
    """Inputs, output buffers and the context (or batch) a program keeps; released with the object."""

    def __init__(self):
        self.ctx = self.batch = None

    def __del__(self):
        if self.ctx is not None:
            dgp.dgp_destroy(self.ctx)
        if self.batch is not None:
            dgp.dgp_batch_destroy(self.batch)


def _parts(x, p):
    return dgp.particles(x[0], x[1], x[2], p[0], p[1], p[2])


def prepare(case, seed):
    s = State()
    s.case, s.inp = case, _inputs(case, seed)
    kind, t = case["kind"], _dtype(case)
    # runs use a stream of their own, as a program that overlaps other work does; some calls the default one
    s.stream = torch.cuda.Stream() if case.get("side", True) else torch.cuda.default_stream()
    torch.cuda.synchronize()
    if kind == "batch":
        m = _members(case)
        s.batch, s.ctxs = dgp.dgp_batch_create(
            [dgp.params(box, n, rc, precision=PRECISION[case["prec"]], tol=_tol(case)) for n, box, rc in m], OM)
        s.box = [box for _, box, _ in m]
        s.x, s.p = [torch.empty_like(v) for v in s.inp["x"]], [torch.empty_like(v) for v in s.inp["p"]]
        s.parts = [_parts(x, p) for x, p in zip(s.x, s.p)]
        return s
    n = case["n"]
    s.ctx = dgp.dgp_init(case["box"], n, case.get("rc", 1.0), OM, precision=PRECISION[case["prec"]], tol=_tol(case),
                         stream=s.stream.cuda_stream)
    if kind == "solve":
        s.out = [torch.empty((n, n, n), dtype=t, device="cuda") for _ in range(4)]
    elif kind in ("steps", "snapshot"):
        s.x, s.p = torch.empty_like(s.inp["x"]), torch.empty_like(s.inp["p"])
        s.parts = _parts(s.x, s.p)
        if kind == "snapshot":
            s.cells = torch.empty(n ** 3 + 1, dtype=torch.int32, device="cuda")
            s.delta = torch.empty((n, n, n), dtype=t, device="cuda")
    elif kind == "adjoint":
        s.start = _parts(s.inp["x"], s.inp["p"])
        s.xb, s.pb = torch.empty_like(s.inp["xb"]), torch.empty_like(s.inp["pb"])
        s.cot = _parts(s.xb, s.pb)
    elif kind == "zeldovich":
        s.x = torch.empty((3, n ** 3), dtype=t, device="cuda")
        s.p = torch.empty_like(s.x)
        s.parts, s.cot = _parts(s.x, s.p), _parts(s.inp["xb"], s.inp["pb"])
        s.grad = torch.empty((n, n, n), dtype=t, device="cuda")
        lat = (torch.arange(n, device="cuda").double() * (case["box"] / n)).to(t)
        s.q = torch.stack([v.reshape(-1) for v in torch.meshgrid(lat, lat, lat, indexing="ij")])
    torch.cuda.synchronize()
    return s


def _unwrap(x, x0, box):
    return x + box * torch.round((x0 - x) / box)


def _spectrum(v, case):
    """A spectrum kept in the type of the mesh it was measured on."""
    return torch.from_numpy(np.ascontiguousarray(v)).to(_dtype(case))


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "batch":
        sched = _schedule(c)
        for x, p, x0, p0 in zip(s.x, s.p, s.inp["x"], s.inp["p"]):
            x.copy_(x0)
            p.copy_(p0)
        for ctx in s.ctxs:
            dgp.dgp_reset(ctx)
        k = len(s.x)
        for a, a1 in zip(sched, sched[1:]):
            dgp.dgp_batch_step(s.batch, s.parts, [a] * k, [a1 - a] * k)
        out = {}
        for n in (48, 64, 96):  # the realisations of one size as one array
            m = [i for i, x in enumerate(s.x) if x.shape[1] == n ** 3]
            if m:
                out["x%d" % n] = torch.stack([_unwrap(s.x[i], s.inp["x"][i], s.box[i]) for i in m])
                out["p%d" % n] = torch.stack([s.p[i] for i in m])
        return out
    with torch.cuda.stream(s.stream):
        if kind == "solve":
            dgp.dgp_reset(s.ctx)
            dgp.dgp_solve_forces(s.ctx, c["a"], s.inp["delta"], *s.out, _tol(c))
            return {"phi": s.out[0], "g": s.out[1:]}
        if kind == "steps":
            s.x.copy_(s.inp["x"])
            s.p.copy_(s.inp["p"])
            dgp.dgp_reset(s.ctx)
            sched = _schedule(c)
            for a, a1 in zip(sched, sched[1:]):
                dgp.pm_step(s.ctx, s.parts, a, a1 - a)
            return {"x": _unwrap(s.x, s.inp["x"], c["box"]), "p": s.p}
        if kind == "adjoint":
            s.xb.copy_(s.inp["xb"])
            s.pb.copy_(s.inp["pb"])
            dgp.dgp_reset(s.ctx)
            a, a1 = _schedule(c)
            dgp.pm_step_adjoint(s.ctx, s.start, a, a1 - a, s.cot)
            return {"xb": s.xb, "pb": s.pb}
        if kind == "zeldovich":
            vf = _velocity_factor(c["a"], 1.0)
            dgp.dgp_zeldovich(s.ctx, s.inp["delta"], vf, s.parts)
            dgp.dgp_zeldovich_adjoint(s.ctx, s.cot, vf, s.grad)
            return {"x": _unwrap(s.x, s.q, c["box"]), "p": s.p, "grad": s.grad}
        if kind == "snapshot":
            s.x.copy_(s.inp["x"])
            s.p.copy_(s.inp["p"])
            # the order inside a cell is not specified, so the permuted arrays show in the cells and the density
            dgp.dgp_sort_particles(s.ctx, s.parts, s.cells)
            dgp.dgp_deposit(s.ctx, s.parts, s.delta)
            k, pk, modes = dgp.power_spectrum(s.ctx, s.delta, c["n"] // 2)
            return {"cells": s.cells, "delta": s.delta, "k": _spectrum(k, c), "pk": _spectrum(pk, c), "modes": modes}
        theta = _angles(c)
        b, q = dgp.bispectrum(s.ctx, s.inp["delta"], c["k1"], c["k2"], theta)
        return {"b": _spectrum(b, c), "q": _spectrum(q, c)}


def _angles(c):
    return [math.pi * (0.05 + 0.9 * i / max(1, c["nth"] - 1)) for i in range(c["nth"])]


def work(case):
    """Inputs and outputs once, and the transforms of the field solves: a real 3D transform is 2.5 m log2 m
    operations, seven of them and about 40 operations a point for each residual evaluation, taken as 15 a solve."""
    b = 8.0 if case["prec"] == "fp64" else 4.0

    def fft(n):
        return 2.5 * n ** 3 * math.log2(n ** 3)

    def solve(n):
        return 15 * (7 * fft(n) + 40.0 * n ** 3) + 6 * fft(n)

    kind = case["kind"]
    if kind == "batch":
        k = case["steps"] + 1
        return {"bytes": sum(12 * b * n ** 3 for n, _, _ in _members(case)),
                "flops": sum(k * solve(n) for n, _, _ in _members(case))}
    n = case["n"]
    m = float(n) ** 3
    if kind == "solve":
        return {"bytes": 5 * b * m, "flops": solve(n)}
    if kind == "steps":
        return {"bytes": 12 * b * m, "flops": (case["steps"] + 1) * solve(n)}
    if kind == "adjoint":
        return {"bytes": 18 * b * m, "flops": 5 * solve(n)}
    if kind == "zeldovich":
        return {"bytes": 14 * b * m, "flops": 8 * fft(n)}
    if kind == "snapshot":
        return {"bytes": 12 * b * case["np"] + (4 + b) * m, "flops": 80.0 * case["np"] + fft(n)}
    return {"bytes": b * m + 16.0 * case["nth"], "flops": (2 + case["nth"]) * 2 * fft(n)}


# ---------------------------------------------------------------------------- the method in 64 bits
def _hubble(a, rc):
    e = 1.0 / rc
    return 0.5 * (e + math.sqrt(e * e + 4.0 * OM * a ** -3))


def _time_integral(a0, a1, rc, power):
    """int dlna / (a^power E) by 8-point Gauss-Legendre."""
    t, w = np.polynomial.legendre.leggauss(8)
    l0, l1 = math.log(a0), math.log(a1)
    x = 0.5 * (l0 + l1) + 0.5 * (l1 - l0) * t
    return 0.5 * (l1 - l0) * float(sum(wi / (math.exp(power * xi) * _hubble(math.exp(xi), rc)) for wi, xi in zip(w, x)))


def _rfft(f):
    return torch.fft.rfftn(f)


def _irfft(f, n):
    return torch.fft.irfftn(f, s=(n, n, n))


class Field:
    """Fourier multipliers and coefficients of the field equations at one scale factor."""

    def __init__(self, n, box, a, rc):
        self.n = n
        self.k, self.q = _axes(n, box)
        self.k2 = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        self.k2[0, 0, 0] = 1.0
        E = _hubble(a, rc)
        eta = rc * E
        den = eta * (2 * eta - 1)
        self.alpha = 3 * (2 * eta * eta - 2 * eta + 1) / den
        self.beta = (2 * eta * eta - 2 * eta - 1) / den
        self.s = 3 * (eta - 1) / eta
        self.c2 = 3 * self.beta * (eta - 1) / (2 * eta - 1)
        self.c3 = (3 * eta * eta - 5 * eta + 1) / (2 * eta * eta * (2 * eta - 1))
        self.eta, self.aE = eta, a * E
        self.ikb = self.aE / CH / torch.sqrt(self.k2)
        self.pairs = [(0, 0), (1, 1), (0, 1), (0, 2), (1, 2)]

    def hess(self, f, i, j):
        v = self.k[i] * self.k[j]
        if i != j:
            v = torch.where(self.q[i] | self.q[j], v.abs(), v)
        return _irfft(f * (v / self.k2), self.n)

    def terms(self, D):
        """Mean-free D, its spectrum and second derivatives xx, yy, xy, xz, yz, zz."""
        f = _rfft(D)
        f[0, 0, 0] = 0
        D = _irfft(f, self.n)
        h = [self.hess(f, i, j) for i, j in self.pairs]
        h.append(D - h[0] - h[1])
        return D, f, h

    def rest(self, D, f, h, S):
        """R of the field equation (c2 N = -c2 D / kbar in Fourier space)."""
        q = D * D - h[0] ** 2 - h[1] ** 2 - h[5] ** 2 - 2 * (h[2] ** 2 + h[3] ** 2 + h[4] ** 2)
        return q + self.alpha * D - self.c2 * _irfft(f * self.ikb, self.n) - S

    def solve(self, delta, tol, start=None):
        """(delta(k), D, D(k), second derivatives) of the converged equation."""
        dk = _rfft(delta)
        dk[0, 0, 0] = 0
        sk = self.s * (1 - self.beta * self.ikb) * dk
        S = _irfft(sk, self.n)
        eps = S.abs().mean().item()
        D = _irfft(sk / (self.alpha - self.c2 * self.ikb), self.n) if start is None else start
        del sk
        best = (math.inf,)
        for it in range(400):
            D, f, h = self.terms(D)
            R = self.rest(D, f, h, S)
            r = R.abs().mean().item() / eps
            if r < best[0]:
                best = (r, D, f, h, it)
            if r < tol or it - best[4] >= 10:
                break
            B = D * ((1 - W) * D + self.alpha) - R
            disc = (self.alpha ** 2 + 4 * (1 - W) * B).clamp_min(0.0)
            D = (torch.sqrt(disc) - self.alpha) / (2 * (1 - W))
            del R, B, disc, h, f
        return dk, best[1], best[2], best[3]

    def phi_k(self, dk, f):
        om = (self.eta - 1) / self.eta
        v = (1.5 * om * dk + f * (self.c3 * self.ikb - 0.5 / self.eta)) * (-self.aE ** 2 / self.k2)
        v = v / (1 + self.ikb / self.eta)
        v[0, 0, 0] = 0
        return v

    def grad(self, f, i, sign=-1.0):
        return torch.where(self.q[i], 0.0, sign * 1j * self.k[i]) * f

    def forces(self, dk, f):
        p = self.phi_k(dk, f)
        return p, [_irfft(self.grad(p, i), self.n) for i in range(3)]

    def adjoint(self, D, h, gbar, tol):
        """delta cotangent for force cotangents gbar, D and h those of the converged solve."""
        n = self.n
        pb = sum(self.grad(_rfft(gbar[i]), i, 1.0) for i in range(3))  # transpose of -i k is +i k
        om = (self.eta - 1) / self.eta
        pref = -self.aE ** 2 / self.k2 / (1 + self.ikb / self.eta)
        pb[0, 0, 0] = 0
        A, B = 1.5 * om * pref * pb, (self.c3 * self.ikb - 0.5 / self.eta) * pref * pb
        g = _irfft(B, n)
        diag = 2 * (1 - W) * D + self.alpha
        weight = [(0, 0, h[0]), (1, 1, h[1]), (2, 2, h[5])] + [(i, j, 2 * v) for (i, j), v in zip(self.pairs[2:], h[2:5])]
        scale = g.abs().mean().item()

        def other(lam):
            f = _rfft(lam)
            f[0, 0, 0] = 0
            acc = self.c2 * self.ikb * f
            for i, j, v in weight:
                m = self.k[i] * self.k[j]
                if i != j:
                    m = torch.where(self.q[i] | self.q[j], m.abs(), m)
                acc = acc + 2 * (m / self.k2) * _rfft(v * lam)
            acc[0, 0, 0] = 0
            return 2 * W * D * lam - _irfft(acc, n)

        def mean_free(rhs):
            return (rhs - (rhs / diag).mean() / (1 / diag).mean()) / diag

        lam = mean_free(g)
        for _ in range(400):
            o = other(lam)
            r = diag * lam + o - g
            if (r - r.mean()).abs().mean().item() < tol * scale:
                break
            lam = mean_free(g - o)
        lk = _rfft(lam)
        lk[0, 0, 0] = 0
        return _irfft(A + self.s * (1 - self.beta * self.ikb) * lk, n)


def _corners(x, n, box):
    """Flat mesh index and CIC weight of the eight corners; the weights carry the gradient of x."""
    u = x.double() * (n / box)
    lo = torch.floor(u.detach())
    f = u - lo
    lo = torch.remainder(lo.long(), n)
    for c in range(8):
        b = [(c >> 2) & 1, (c >> 1) & 1, c & 1]
        j = [torch.remainder(lo[i] + b[i], n) for i in range(3)]
        w = [f[i] if b[i] else 1 - f[i] for i in range(3)]
        yield (j[0] * n + j[1]) * n + j[2], w[0] * w[1] * w[2]


def _deposit(x, n, box):
    rho = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    for i, w in _corners(x, n, box):
        rho = rho.index_add(0, i, w)
    return (rho * (n ** 3 / x.shape[1]) - 1.0).reshape(n, n, n)


def _gather(g, x, n, box):
    out = 0
    for i, w in _corners(x, n, box):
        out = out + w * torch.stack([v.reshape(-1)[i] for v in g])
    return out


def _exact_steps(x, p, n, box, rc, sched, tol):
    x0 = x.double()
    x, p, D, F = x.double(), p.double(), None, None
    for a, a1 in zip(sched, sched[1:]):
        ah = math.sqrt(a * a1)

        def force(x, a, D):
            fld = Field(n, box, a, rc)
            dk, D, f, _ = fld.solve(_deposit(x, n, box), tol, D)
            return D, _gather(fld.forces(dk, f)[1], x, n, box)

        if F is None:
            D, F = force(x, a, D)
        p = p + _time_integral(a, ah, rc, 0) * F
        x = x + _time_integral(a, a1, rc, 2) * p
        D, F = force(torch.remainder(x, box), a1, D)
        p = p + _time_integral(ah, a1, rc, 0) * F
    return x + box * torch.round((x0 - x) / box), p


def _force_vjp(x, fbar, n, box, a, rc, tol):
    """sum fbar . dF/dx for the particle forces F(x): through the gather, the solve and the deposit."""
    x = x.detach().clone().requires_grad_(True)
    delta = _deposit(x, n, box)
    with torch.no_grad():
        fld = Field(n, box, a, rc)
        dk, D, f, h = fld.solve(delta.detach(), tol)
        g = fld.forces(dk, f)[1]
    g = [v.requires_grad_(True) for v in g]
    gb = torch.autograd.grad((_gather(g, x, n, box) * fbar).sum(), g + [x])
    db = fld.adjoint(D, h, gb[:3], tol)
    return gb[3] + torch.autograd.grad(delta, x, db)[0]


def exact(case, seed):
    inp, kind = _inputs(case, seed), case["kind"]
    tol = 1e-13 if case["prec"] == "fp64" else 1e-9
    if kind == "batch":
        out = {}
        for (n, box, rc), x, p in zip(_members(case), inp["x"], inp["p"]):
            for name, v in zip("xp", _exact_steps(x, p, n, box, rc, _schedule(case), tol)):
                out.setdefault("%s%d" % (name, n), []).append(v)
        return {k: torch.stack(v) for k, v in out.items()}
    n, box = case["n"], case["box"]
    if kind == "solve":
        fld = Field(n, box, case["a"], case["rc"])
        dk, _, f, _ = fld.solve(inp["delta"].double(), tol)
        p, g = fld.forces(dk, f)
        return {"phi": _irfft(p, n), "g": g}
    if kind == "steps":
        x, p = _exact_steps(inp["x"], inp["p"], n, box, case["rc"], _schedule(case), tol)
        return {"x": x, "p": p}
    if kind == "adjoint":
        rc = case["rc"]
        a, a1 = _schedule(case)
        ah = math.sqrt(a * a1)
        x0, xb, pb = inp["x"].double(), inp["xb"].double(), inp["pb"].double()
        k1, dr, k2 = _time_integral(a, ah, rc, 0), _time_integral(a, a1, rc, 2), _time_integral(ah, a1, rc, 0)
        with torch.no_grad():
            fld = Field(n, box, a, rc)
            dk, _, f, _ = fld.solve(_deposit(x0, n, box), tol)
            ph = inp["p"].double() + k1 * _gather(fld.forces(dk, f)[1], x0, n, box)
            x1 = torch.remainder(x0 + dr * ph, box)
        xb = xb + _force_vjp(x1, k2 * pb, n, box, a1, rc, tol)
        pb = pb + dr * xb
        xb = xb + _force_vjp(x0, k1 * pb, n, box, a, rc, tol)
        return {"xb": xb, "pb": pb}
    if kind == "zeldovich":
        vf = _velocity_factor(case["a"], 1.0)
        fld = Field(n, box, 1.0, 1.0)
        dk = _rfft(inp["delta"].double())
        dk[0, 0, 0] = 0
        psi = torch.stack([_irfft(fld.grad(dk / fld.k2, i, 1.0), n).reshape(-1) for i in range(3)])
        lat = torch.arange(n, device="cuda").double() * (box / n)
        q = torch.stack([v.reshape(-1) for v in torch.meshgrid(lat, lat, lat, indexing="ij")])
        cot = inp["xb"].double() + vf * inp["pb"].double()
        acc = sum(fld.grad(_rfft(cot[i].reshape(n, n, n)) / fld.k2, i, -1.0) for i in range(3))
        acc[0, 0, 0] = 0
        return {"x": q + psi, "p": vf * psi, "grad": _irfft(acc, n)}
    kf = 2.0 * math.pi / box
    if kind == "snapshot":
        delta = _deposit(inp["x"], n, box)
        f = _rfft(delta)
        k, _ = _axes(n, box)
        km = torch.sqrt(k[0] ** 2 + k[1] ** 2 + k[2] ** 2)
        w = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device="cuda")
        w[0] = w[-1] = 1.0
        w = w.expand(n, n, n // 2 + 1).reshape(-1)
        b = torch.floor(km / kf + 0.5).long().reshape(-1)
        b = torch.where(b > n // 2, torch.zeros_like(b), b)

        def shell(v):
            return torch.zeros(n // 2 + 1, dtype=torch.float64, device="cuda").index_add(0, b, w * v.reshape(-1))[1:]

        cnt = shell(torch.ones_like(w))
        pk = shell(box ** 3 * (f.real ** 2 + f.imag ** 2) / float(n) ** 6) / cnt
        return {"cells": None, "delta": delta, "k": shell(km) / cnt, "pk": pk, "modes": None}
    # bispectrum: shells of width k_f around k1, k2 and |k1 + k2|
    m3 = float(n) ** 3
    f = _rfft(inp["delta"].double())
    f[0, 0, 0] = 0
    k, _ = _axes(n, box)
    km = torch.sqrt(k[0] ** 2 + k[1] ** 2 + k[2] ** 2) / kf
    one = torch.ones_like(f)

    def shells(kc):
        sel = (km > (kc - 0.5 * kf) / kf) & (km < (kc + 0.5 * kf) / kf) & (km > 0)
        return _irfft(f * sel, n), _irfft(one * sel, n)

    def power(d, i):
        return box ** 3 / m3 ** 2 * ((d * d).sum() / (i * i).sum())

    d1, i1 = shells(case["k1"])
    d2, i2 = shells(case["k2"])
    P1, P2 = power(d1, i1), power(d2, i2)
    b, q = [], []
    for th in _angles(case):
        d3, i3 = shells(math.sqrt(case["k1"] ** 2 + case["k2"] ** 2 + 2 * case["k1"] * case["k2"] * math.cos(th)))
        P3 = power(d3, i3)
        b.append(box ** 6 / m3 ** 3 * (d1 * d2 * d3).sum() / (i1 * i2 * i3).sum())
        q.append(b[-1] / (P1 * P2 + P2 * P3 + P3 * P1))
    return {"b": torch.stack(b), "q": torch.stack(q)}
