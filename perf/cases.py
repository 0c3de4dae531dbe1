"""Performance cases: the evaluations, flow steps and training passes a user of the library runs.

A case is a dict of plain values; `prepare` builds what a program holds before the call (the
plan, batch or network handle and the device inputs), `run` makes one pass through the public
entry points, `exact` gives the same outputs from plain 64-bit torch.

Kinds: "eval3d", "eval2d", "eval1d" (one potential evaluation of a plan), "batch" (several FP32
plans evaluated by one call), "gf" (one gradient-flow step), "ts" (one time step of the
dynamics), "net" (loss and gradients of the initial-guess network).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1410_3584_gb300 as nl

NET_GRID = 48
NET_BOX = 10.0


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # smallest 3D evaluation in use: the paper's closed-form check (rho = exp(-|x|^2) on
        # [-8,8)^3, 32 x 32 x 64 nodes); launches and latency count
        dict(name="coulomb3d_32_fp64", kind="eval3d", kernel="coulomb3d", prec="fp64", method=0, nx=32, ny=32, nz=32,
             Lx=8.0, Ly=8.0, Lz=8.0, ax=1.0, ay=1.0, az=1.0, peps=1e16, tol=1e-12, nr=32, nth=32, nph=64),
        # the headline workload in single precision: anisotropic Gaussian, 128^3 over [-12,12)^3
        dict(name="coulomb3d_128_fp32", kind="eval3d", kernel="coulomb3d", prec="fp32", method=0, nx=128, ny=128,
             nz=128, Lx=12.0, Ly=12.0, Lz=12.0, ax=1.0, ay=math.sqrt(2.0), az=2.0, peps=1e16, tol=1e-6),
        # the same density in double precision with the dipolar kernel (axis z): the largest case
        dict(name="dipole3d_128_fp64", kind="eval3d", kernel="dipole3d", prec="fp64", method=0, nx=128, ny=128,
             nz=128, Lx=12.0, Ly=12.0, Lz=12.0, ax=1.0, ay=math.sqrt(2.0), az=2.0, peps=1e16, tol=1e-12),
        # an ordinary trap shape: uneven box with radix-3 and radix-5 lengths, tilted dipole axis
        dict(name="dipole3d_90x64x108_fp32", kind="eval3d", kernel="dipole3d", prec="fp32", method=0, nx=90, ny=64,
             nz=108, Lx=8.0, Ly=6.0, Lz=10.0, ax=1.3, ay=1.0, az=1.6, peps=1e8, tol=1e-6, dx=1.0, dy=0.5, dz=1.0),
        # the improved algorithm (small-ball NUFFT plus FFT convolution) in double precision
        dict(name="split3d_96_fp64", kind="eval3d", kernel="coulomb3d", prec="fp64", method=2, nx=96, ny=96, nz=96,
             Lx=10.0, Ly=10.0, Lz=10.0, ax=1.0, ay=1.2, az=1.5, peps=1e16, tol=1e-12),
        # 2D Coulomb on 1024^2 over [-16,16)^2, three Gaussians, single precision
        dict(name="coulomb2d_1024_fp32", kind="eval2d", kernel="coulomb2d", prec="fp32", method=0, nx=1024, ny=1024,
             Lx=16.0, Ly=16.0, amin=0.5, peps=1e16, tol=1e-6),
        # 2D Poisson (near-origin correction) on an uneven grid, double precision
        dict(name="poisson2d_640x768_fp64", kind="eval2d", kernel="poisson2d", prec="fp64", method=0, nx=640, ny=768,
             Lx=16.0, Ly=16.0, amin=0.5, peps=1e16, tol=1e-12),
        # 1D Poisson, the smallest path of the library
        dict(name="poisson1d_1024_fp64", kind="eval1d", kernel="poisson1d", prec="fp64", nx=1024, Lx=16.0, amin=0.5),
        # several densities on uneven grids with mixed kernels in one call
        dict(name="batch_8_mixed_fp32", kind="batch", count=8, sizes="64,96,128,160", spec=20141014, form="graph",
             branches=8),
        # one ground-state step (dipolar plus contact term) on 96^3 over [-10,10)^3 with the
        # precomputed kernel, the plan the ground-state solver uses
        dict(name="gf_dipole_96_fp64", kind="gf", kernel="dipole3d", method=1, n=96, L=10.0, beta=50.0, g=100.0,
             gamma=2.0, tau=1e-2, inner_tol=1e-12),
        # one fourth-order step of the 3D dynamics (h = 1/4 on [-8,8)^3)
        dict(name="ts_coulomb_64_fp64", kind="ts", kernel="coulomb3d", prec="fp64", method=1, n=64, L=8.0, beta=5.0,
             g=0.0, tau=1e-3, order=4),
        # training pass of the initial-guess network at the batch the ground-state workload uses
        dict(name="net_gradients_64", kind="net", batch=64),
    ]


def _good(lo, hi):
    out = []
    for n in range(lo + lo % 2, hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _log_pick(rng, lo, hi):
    """An even 2-3-5 length between lo and hi, spread over the logarithm of the range."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(_good(lo, hi), key=lambda n: abs(n - t))


def draw(rng):
    kind = rng.choice(["eval3d"] * 6 + ["eval2d"] * 3 + ["eval1d", "batch", "gf", "ts", "net"])
    if kind == "eval3d":
        prec = rng.choice(["fp32", "fp64"])
        method = rng.choice([0, 0, 0, 1, 2])
        hi = 192 if prec == "fp32" and method == 0 else 128
        n = _log_pick(rng, 24, hi)
        ns = [n] * 3 if rng.random() < 0.4 else [max(24, _log_pick(rng, max(24, n // 2), n)) for _ in range(3)]
        rng.shuffle(ns)
        a = [round(rng.uniform(1.0, 1.6), 3) for _ in range(3)]
        tol = rng.choice([1e-6, 1e-6, 1e-6, 1e-5, 1e-4]) if prec == "fp32" else rng.choice([1e-12, 1e-12, 1e-10])
        c = dict(kind=kind, kernel=rng.choice(["coulomb3d", "dipole3d"]), prec=prec, method=method, nx=ns[0],
                 ny=ns[1], nz=ns[2], Lx=6 * a[0], Ly=6 * a[1], Lz=6 * a[2], ax=a[0], ay=a[1], az=a[2],
                 peps=1e16 if prec == "fp64" else rng.choice([1e8, 1e16]), tol=tol)
        if c["kernel"] == "dipole3d" and rng.random() < 0.5:
            c.update(dx=rng.uniform(-1, 1), dy=rng.uniform(-1, 1), dz=1.0)
        return c
    if kind == "eval2d":
        kernel = rng.choice(["coulomb2d", "poisson2d"])
        nx = _log_pick(rng, 64, 1024)
        ny = nx if rng.random() < 0.4 else _log_pick(rng, max(64, nx // 2), min(1024, 2 * nx))
        return dict(kind=kind, kernel=kernel, prec=rng.choice(["fp32", "fp64"]), method=rng.choice([0, 0, 2]), nx=nx,
                    ny=ny, Lx=16.0, Ly=16.0, amin=round(rng.uniform(0.5, 1.0), 3), peps=1e16, tol=0.0)
    if kind == "eval1d":
        return dict(kind=kind, kernel="poisson1d", prec="fp64", nx=_log_pick(rng, 128, 1024), Lx=16.0, amin=0.5)
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 8), sizes="64,96,128", spec=rng.randint(1, 10 ** 6),
                    form=rng.choice(["graph", "graph", "persistent"]), branches=rng.choice([1, 4, 8]))
    if kind == "gf":
        kernel = rng.choice(["coulomb3d", "dipole3d"])
        beta = math.exp(rng.uniform(0.0, math.log(200.0)))
        return dict(kind=kind, kernel=kernel, method=rng.choice([1, 1, 2]), n=_log_pick(rng, 48, 96), L=10.0,
                    beta=beta if kernel == "coulomb3d" else 0.5 * beta, g=0.0 if kernel == "coulomb3d" else beta,
                    gamma=rng.uniform(1.0, 4.0), tau=1e-2, inner_tol=1e-12)
    if kind == "ts":
        return dict(kind=kind, kernel=rng.choice(["coulomb3d", "dipole3d"]), prec=rng.choice(["fp64", "fp64", "fp32"]),
                    method=rng.choice([1, 1, 0, 2]), n=_log_pick(rng, 32, 64), L=8.0, beta=rng.uniform(1.0, 20.0),
                    g=rng.choice([0.0, 2.0]), tau=1e-3, order=rng.choice([2, 4]))
    return dict(kind=kind, batch=rng.randint(1, 128))


# ------------------------------------------------------------------ inputs
def _dtype(prec):
    return torch.float64 if prec == "fp64" else torch.float32


def _axes(n, L):
    return [torch.arange(m, dtype=torch.float64, device="cuda") * (2.0 * l / m) - l for m, l in zip(n, L)]


def _gauss(n, L, a, c, amp):
    """amp exp(-sum (x - c)^2 / a^2) on the grid (x_m = -L + m h, C order), 64 bits."""
    out = torch.full((), float(amp), dtype=torch.float64, device="cuda")
    for d, x in enumerate(_axes(n, L)):
        e = torch.exp(-((x - c[d]) / a[d]) ** 2)
        out = out.unsqueeze(-1) * e
    return out


def _radius(L, n, a_min, peps):
    """Truncation radius of the Fourier ball: where the Gaussian's transform falls below 1/peps."""
    return min(math.pi / max(2.0 * l / m for l, m in zip(L, n)), 2.0 * math.sqrt(math.log(peps)) / a_min)


def _rho3(case, seed):
    n, L = (case["nx"], case["ny"], case["nz"]), (case["Lx"], case["Ly"], case["Lz"])
    a = (case["ax"], case["ay"], case["az"])
    r = np.random.default_rng(seed)
    rho = 0.0
    for amp in r.uniform(0.5, 1.5, 2):
        rho = rho + _gauss(n, L, a, r.uniform(-0.4, 0.4, 3) * np.array(a), amp)
    return rho.to(_dtype(case["prec"])).contiguous()


def _mix(case, seed, dim):
    """Three Gaussians: centres in [-4,4]^d, widths in [amin, 2], amplitudes in [0.5, 1.5]."""
    r = np.random.default_rng(seed)
    return [(r.uniform(-4, 4, dim), float(r.uniform(case["amin"], 2.0)), float(r.uniform(0.5, 1.5))) for _ in range(3)]


def _rho_mix(case, seed, n, L):
    rho = sum(_gauss(n, L, [s] * len(n), c, amp) for c, s, amp in _mix(case, seed, len(n)))
    return rho.to(_dtype(case["prec"])).contiguous()


def _batch_items(case):
    """Per item: n from the sizes, widths (1, r, r) with r in [1, 4], box 6 times the largest."""
    r = np.random.default_rng(case["spec"])
    sizes = [int(s) for s in case["sizes"].split(",")]
    items = []
    for _ in range(case["count"]):
        n = int(r.choice(sizes))
        a = (1.0, float(r.uniform(1, 4)), float(r.uniform(1, 4)))
        items.append((n, 6.0 * max(a), a, "coulomb3d" if r.uniform() < 0.5 else "dipole3d"))
    return items


def _batch_rho(item, seed):
    n, L, a, _ = item
    r = np.random.default_rng(seed)
    return _gauss((n,) * 3, (L,) * 3, a, r.uniform(-0.3, 0.3, 3), r.uniform(0.5, 1.5)).float().contiguous()


def _trap(n, L, gamma):
    x, y, z = _axes((n,) * 3, (L,) * 3)
    return (0.5 * (x[:, None, None] ** 2 + y[None, :, None] ** 2 + (gamma * z[None, None, :]) ** 2)).contiguous()


def _gf_start(case, seed):
    n, L = case["n"], case["L"]
    r = np.random.default_rng(seed)
    s = math.sqrt(2.0) * r.uniform(0.9, 1.5)
    phi = _gauss((n,) * 3, (L,) * 3, (s, s, s / math.sqrt(case["gamma"])), r.uniform(-0.2, 0.2, 3), 1.0)
    return (phi / torch.sqrt((2.0 * L / n) ** 3 * (phi * phi).sum())).contiguous()


def _ts_start(case, seed):
    n, L = case["n"], case["L"]
    r = np.random.default_rng(seed)
    amp = _gauss((n,) * 3, (L,) * 3, math.sqrt(2.0) * r.uniform(0.9, 1.1, 3), r.uniform(-0.3, 0.3, 3), 1.0)
    k = r.uniform(-1, 1, 3)
    ph = sum(float(k[d]) * x.reshape([-1 if e == d else 1 for e in range(3)]) for d, x in enumerate(_axes((n,) * 3, (L,) * 3)))
    return torch.polar(amp, ph).to(torch.complex128 if case["prec"] == "fp64" else torch.complex64).contiguous()


_NET_DENSE = ((64, 512), (512, 512), (512, 512), (512, 512), (512, 1792))
_NET_CONV = ((8, 8), (8, 8), (8, 1))


def _net_params(seed):
    """The flat parameter vector: uniform weights in +-1/sqrt(fan in), zero biases, zero padding."""
    r = np.random.default_rng(seed)
    out = []
    for l, (ni, no) in enumerate(_NET_DENSE):
        w = np.zeros((no, ni), dtype=np.float32)
        rows, cols = (1728 if l == 4 else no), (4 if l == 0 else ni)
        w[:rows, :cols] = r.uniform(-1, 1, (rows, cols)) / math.sqrt(cols)
        out += [w.ravel(), np.zeros(no, dtype=np.float32)]
    for ci, co in _NET_CONV:
        out += [(r.uniform(-1, 1, co * ci * 27) / math.sqrt(27 * ci)).astype(np.float32), np.zeros(co, dtype=np.float32)]
    return np.concatenate(out)


def _net_inputs(case, seed):
    """Features of random ground-state problems and smooth bumps on the cube as targets."""
    r = np.random.default_rng(seed + 7)
    B = case["batch"]
    f = np.stack([r.uniform(0, 1, B), r.uniform(0, 1, B), np.zeros(B), np.zeros(B)], 1)
    k = r.integers(0, 2, B)
    f[np.arange(B), 2 + k] = 1.0
    x = torch.arange(NET_GRID, dtype=torch.float32, device="cuda") * (2 * NET_BOX / NET_GRID) - NET_BOX
    s = torch.from_numpy(r.uniform(1.0, 3.0, (B, 3)).astype(np.float32)).cuda()
    e = torch.exp(-(x[None, None, :] / s[:, :, None]) ** 2)
    amp = torch.from_numpy(r.uniform(-0.3, 0.1, B).astype(np.float32)).cuda()
    t = amp[:, None, None, None] * e[:, 0, :, None, None] * e[:, 1, None, :, None] * e[:, 2, None, None, :]
    return torch.from_numpy(f.astype(np.float32)).cuda(), t.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "eval3d":
        n, L = (case["nx"], case["ny"], case["nz"]), (case["Lx"], case["Ly"], case["Lz"])
        counts = (case["nr"], case["nth"], case["nph"]) if "nr" in case else None
        P = _radius(L, n, min(case["ax"], case["ay"], case["az"]), case["peps"])
        axis = (case.get("dx", 0.0), case.get("dy", 0.0), case.get("dz", 1.0))
        s["plan"] = nl.Plan(n, L, case["kernel"], case["prec"], kmax=P, counts=counts, tol=case["tol"],
                            method=case["method"], dipole_axis=axis)
        s["rho"] = _rho3(case, seed)
    elif kind == "eval2d":
        n, L = (case["nx"], case["ny"]), (case["Lx"], case["Ly"])
        s["plan"] = nl.Plan(n, L, case["kernel"], case["prec"], kmax=_radius(L, n, case["amin"], case["peps"]),
                            tol=case["tol"], method=case["method"])
        s["rho"] = _rho_mix(case, seed, n, L)
    elif kind == "eval1d":
        s["plan"] = nl.Plan((case["nx"],), (case["Lx"],), case["kernel"], case["prec"])
        s["rho"] = _rho_mix(case, seed, (case["nx"],), (case["Lx"],))
    elif kind == "batch":
        s["stream"] = torch.cuda.Stream()
        s["items"] = _batch_items(case)
        s["plans"] = [nl.Plan((n,) * 3, (L,) * 3, k, "fp32", kmax=_radius((L,), (n,), 1.0, 1e8), tol=1e-6,
                              dipole_axis=(0.0, 0.0, 1.0), stream=s["stream"]) for n, L, a, k in s["items"]]
        s["rho"] = [_batch_rho(it, seed + i) for i, it in enumerate(s["items"])]
        s["phi"] = [torch.empty_like(r) for r in s["rho"]]
        s["batch"] = nl.nlp_batch_create([p.handle for p in s["plans"]], stream=s["stream"])
        nl.nlp_batch_set_mode(s["batch"], case["form"], case["branches"])
        s["close"] = _Closer(s["batch"], s["plans"])
        torch.cuda.synchronize()
    elif kind == "gf":
        n, L = case["n"], case["L"]
        s["plan"] = nl.Plan((n,) * 3, (L,) * 3, case["kernel"], "fp64", kmax=math.pi * n / (2.0 * L),
                            method=case["method"], dipole_axis=(0.0, 0.0, 1.0))
        s["V"] = _trap(n, L, case["gamma"])
        s["start"] = _gf_start(case, seed)
        s["psi"] = torch.empty_like(s["start"])
    elif kind == "ts":
        n, L = case["n"], case["L"]
        s["plan"] = nl.Plan((n,) * 3, (L,) * 3, case["kernel"], case["prec"], kmax=_radius((L,), (n,), 1.0, 1e16),
                            method=case["method"], dipole_axis=(0.0, 0.0, 1.0))
        s["V"] = _trap(n, L, 1.0).to(_dtype(case["prec"]))
        s["start"] = _ts_start(case, seed)
        s["psi"] = torch.empty_like(s["start"])
    else:
        s["net"] = nl.Surrogate(NET_BOX, 0, 0)
        s["net"].set_params(_net_params(seed))
        s["feat"], s["target"] = _net_inputs(case, seed)
    return s


class _Closer:
    """Destroys the batch handle before the plans it uses."""

    def __init__(self, batch, plans):
        self.batch, self.plans = batch, plans

    def __del__(self):
        nl.nlp_batch_destroy(self.batch)


def run(state):
    kind, case = state["kind"], state["case"]
    if kind in ("eval3d", "eval2d", "eval1d"):
        return state["plan"].eval(state["rho"])
    if kind == "batch":
        state["stream"].wait_stream(torch.cuda.current_stream())
        nl.nlp_batch_eval(state["batch"], state["rho"], state["phi"])
        torch.cuda.current_stream().wait_stream(state["stream"])
        return state["phi"]
    if kind == "gf":
        psi = state["psi"].copy_(state["start"])
        change, _, _, _ = nl.nlp_gf_step(state["plan"].handle, psi, state["V"], case["beta"], case["g"], case["tau"],
                                         case["inner_tol"], 400)
        return {"phi": psi, "change": change}
    if kind == "ts":
        psi = state["psi"].copy_(state["start"])
        nl.nlp_ts_step(state["plan"].handle, psi, state["V"], case["beta"], case["g"], case["tau"], case["order"])
        return psi
    loss, grads = state["net"].gradients(state["feat"], state["target"])
    return {"loss": loss, "grads": grads}


# ------------------------------------------------------------------ floors
def _conv_work(n, size):
    """One aperiodic convolution on the grid: the two real transforms of the doubled grid."""
    N = math.prod(n)
    F = math.prod(2 * m for m in n)
    return 2 * N * size, 2 * 2.5 * F * math.log2(F)


def work(case):
    kind = case["kind"]
    size = 4 if case.get("prec") == "fp32" else 8
    if kind == "eval3d":
        b, f = _conv_work((case["nx"], case["ny"], case["nz"]), size)
    elif kind == "eval2d":
        b, f = _conv_work((case["nx"], case["ny"]), size)
    elif kind == "eval1d":
        b, f = _conv_work((case["nx"],), size)
    elif kind == "batch":
        each = [_conv_work((it[0],) * 3, 4) for it in _batch_items(case)]
        b, f = sum(e[0] for e in each), sum(e[1] for e in each)
    elif kind == "gf":
        N = case["n"] ** 3
        _, f = _conv_work((case["n"],) * 3, 8)
        b, f = 3 * N * 8, f + 2 * 2.5 * N * math.log2(N)       # phi, V in, phi out; one linear solve at least
    elif kind == "ts":
        N, sub = case["n"] ** 3, 1 if case["order"] == 2 else 3
        _, f = _conv_work((case["n"],) * 3, size)
        b, f = (4 + 1) * N * size, sub * (f + 4 * 5 * N * math.log2(N))
    else:
        B = case["batch"]
        dense = 2 * B * sum(i * o for i, o in _NET_DENSE)
        conv = sum(2 * B * 27 * ci * co * g ** 3 for (ci, co), g in zip(_NET_CONV, (12, 24, 48)))
        b, f = 4 * (B * 4 + B * NET_GRID ** 3) + 8 * _net_params(0).size, 3 * (dense + conv)
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------------ 64-bit results
def _fast_len(m):
    return next(n for n in _good(m, 2 * m + 8) if n >= m)


class _Potential3:
    """U * rho on the grid for the 3D Coulomb or dipolar kernel by the truncated-kernel Fourier
    method: (1 - cos R k)/k^2 (the transform of 1/(4 pi r) cut at the box diagonal R) on a grid
    padded past every periodic image; dipolar: 3 (n.k)^2 times that, minus 1."""

    def __init__(self, n, L, kernel, axis=(0.0, 0.0, 1.0)):
        self.n = n
        R = 1.001 * math.sqrt(sum((2 * l) ** 2 for l in L))
        h = [2 * l / m for l, m in zip(L, n)]
        self.pad = [_fast_len(int(math.ceil((2 * l + R) / hh)) + 1) for l, hh in zip(L, h)]
        k = [2 * math.pi * torch.fft.fftfreq(p, d=hh, device="cuda", dtype=torch.float64) for p, hh in zip(self.pad[:2], h)]
        k.append(2 * math.pi * torch.fft.rfftfreq(self.pad[2], d=h[2], device="cuda", dtype=torch.float64))
        kx, ky, kz = k[0][:, None, None], k[1][None, :, None], k[2][None, None, :]
        k2 = kx * kx + ky * ky + kz * kz
        k2[0, 0, 0] = 1.0
        G = 2.0 * torch.sin(0.5 * R * torch.sqrt(k2)) ** 2 / k2
        G[0, 0, 0] = 0.5 * R * R
        self.dip = kernel == "dipole3d"
        if self.dip:
            nn = math.sqrt(sum(a * a for a in axis))
            u = [a / nn for a in axis]
            G = 3.0 * (u[0] * kx + u[1] * ky + u[2] * kz) ** 2 * G
        self.G = G

    def __call__(self, rho):
        rho = rho.double()
        F = torch.fft.rfftn(rho, s=self.pad)
        F *= self.G
        out = torch.fft.irfftn(F, s=self.pad)[:self.n[0], :self.n[1], :self.n[2]]
        return out - rho if self.dip else out.contiguous()


def _ein(z):
    """Ein(z) = int_0^z (1 - e^-t)/t dt = E_1(z) + ln z + gamma: power series up to 2, above it
    the series' value at 2 plus Gauss-Legendre panels doubling in width (to 64), then ln growth."""
    small = torch.clamp(z, max=2.0)
    term, out = torch.ones_like(small), torch.zeros_like(small)
    for k in range(1, 40):
        term = term * (-small / k)
        out = out - term / k
    gx, gw = np.polynomial.legendre.leggauss(24)
    a = 2.0
    while a < 64.0:
        top = torch.clamp(z, min=a, max=2 * a)
        half = 0.5 * (top - a)
        for x, w in zip(gx, gw):
            t = a + half * (1.0 + float(x))
            out = out + float(w) * half * (1.0 - torch.exp(-t)) / t
        a *= 2
    return out + torch.log(torch.clamp(z, min=64.0) / 64.0)


def _exact2(case, seed):
    n, L = (case["nx"], case["ny"]), (case["Lx"], case["Ly"])
    x, y = _axes(n, L)
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    for c, s, amp in _mix(case, seed, 2):
        r2 = (x[:, None] - float(c[0])) ** 2 + (y[None, :] - float(c[1])) ** 2
        if case["kernel"] == "coulomb2d":     # (sqrt(pi) s / 2) e^{-r^2/2s^2} I_0(r^2/2s^2)
            out += amp * 0.5 * math.sqrt(math.pi) * s * torch.special.i0e(r2 / (2 * s * s))
        else:                                 # -(s^2/4) (E_1(r^2/s^2) + ln r^2)
            z = r2 / (s * s)
            out += -amp * 0.25 * s * s * (_ein(z) - 0.57721566490153286061 + 2.0 * math.log(s))
    return out


def _exact1(case, seed):
    x, = _axes((case["nx"],), (case["Lx"],))
    out = torch.zeros_like(x)
    for c, s, amp in _mix(case, seed, 1):
        t = (x - float(c[0])) / s
        out += -amp * 0.5 * s * s * (t * math.sqrt(math.pi) * torch.erf(t) + torch.exp(-t * t))
    return out


def _exact_gf(case, seed):
    n, L, tau = case["n"], case["L"], case["tau"]
    phi, V = _gf_start(case, seed), _trap(n, L, case["gamma"])
    U = _Potential3((n,) * 3, (L,) * 3, case["kernel"])
    rho = phi * phi
    b = V + case["g"] * rho + case["beta"] * U(rho)
    mu = math.pi / L * torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)
    mz = math.pi / L * torch.arange(n // 2 + 1, device="cuda", dtype=torch.float64)
    m2 = mu[:, None, None] ** 2 + mu[None, :, None] ** 2 + mz[None, None, :] ** 2

    def solve(v, alpha):
        return torch.fft.irfftn(torch.fft.rfftn(v) / (1.0 / tau + alpha + 0.5 * m2), s=(n,) * 3)

    # preconditioned conjugate gradients on (1/tau - Delta/2 + b) x = phi/tau
    alpha = 0.5 * float(b.max() + b.min())
    A = lambda v: torch.fft.irfftn(torch.fft.rfftn(v) * (0.5 * m2), s=(n,) * 3) + (1.0 / tau + b) * v  # noqa: E731
    xk = phi.clone()
    r = phi / tau - A(xk)
    z = solve(r, alpha)
    p, rz = z.clone(), (r * z).sum()
    for _ in range(400):
        Ap = A(p)
        a = rz / (p * Ap).sum()
        xk = xk + a * p
        r = r - a * Ap
        z = solve(r, alpha)
        if float(z.abs().max()) < 1e-15:
            break
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    out = xk / torch.sqrt((2.0 * L / n) ** 3 * (xk * xk).sum())
    return {"phi": out, "change": float((out - phi).abs().max()) / tau}


def _exact_ts(case, seed):
    n, L = case["n"], case["L"]
    psi = _ts_start(case, seed).to(torch.complex128)
    V = _trap(n, L, 1.0).to(_dtype(case["prec"])).double()
    U = _Potential3((n,) * 3, (L,) * 3, case["kernel"])
    mu = math.pi / L * torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)
    m2 = mu[:, None, None] ** 2 + mu[None, :, None] ** 2 + mu[None, None, :] ** 2

    def rot(th):
        return torch.polar(torch.ones_like(th), th)

    def strang(v, tau):
        v = torch.fft.ifftn(torch.fft.fftn(v) * rot(-0.25 * tau * m2))
        rho = v.real ** 2 + v.imag ** 2
        v = v * rot(-tau * (V + case["g"] * rho + case["beta"] * U(rho)))
        return torch.fft.ifftn(torch.fft.fftn(v) * rot(-0.25 * tau * m2))

    if case["order"] == 2:
        return strang(psi, case["tau"])
    w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
    for w in (w1, 1.0 - 2.0 * w1, w1):
        psi = strang(psi, w * case["tau"])
    return psi


def _exact_net(case, seed):
    feat, target = _net_inputs(case, seed)
    B = case["batch"]
    p = torch.from_numpy(_net_params(seed)).cuda().double().requires_grad_(True)
    o = 0

    def take(*shape):
        nonlocal o
        m = math.prod(shape)
        v = p[o:o + m].reshape(shape)
        o += m
        return v

    silu = torch.nn.functional.silu
    x = torch.nn.functional.pad(feat.double(), (0, 60))
    for l, (ni, no) in enumerate(_NET_DENSE):
        W, b = take(no, ni), take(no)
        x = x @ W.T + b
        x = silu(x) if l < 4 else x
    z = x[:, :1728].reshape(B, 8, 6, 6, 6)
    for c, (ci, co) in enumerate(_NET_CONV):
        w, b = take(co, ci, 27), take(co)
        z = torch.repeat_interleave(torch.repeat_interleave(torch.repeat_interleave(z, 2, 2), 2, 3), 2, 4)
        g = z.shape[-1]
        zp = torch.nn.functional.pad(z, (1,) * 6)
        y = b.reshape(1, co, 1, 1, 1).expand(B, co, g, g, g)
        for d in range(27):
            dz, dy, dx = d // 9, (d // 3) % 3, d % 3
            y = y + torch.einsum("oi,bizyx->bozyx", w[:, :, d], zp[:, :, dz:dz + g, dy:dy + g, dx:dx + g])
        z = silu(y) if c < 2 else y
    loss = ((z[:, 0] - target.double()) ** 2).mean()
    g, = torch.autograd.grad(loss, p)
    return {"loss": float(loss), "grads": g.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval3d":
        U = _Potential3((case["nx"], case["ny"], case["nz"]), (case["Lx"], case["Ly"], case["Lz"]), case["kernel"],
                        (case.get("dx", 0.0), case.get("dy", 0.0), case.get("dz", 1.0)))
        return U(_rho3(case, seed))
    if kind == "eval2d":
        return _exact2(case, seed)
    if kind == "eval1d":
        return _exact1(case, seed)
    if kind == "batch":
        out = []
        for i, it in enumerate(_batch_items(case)):
            n, L, a, k = it
            out.append(_Potential3((n,) * 3, (L,) * 3, k)(_batch_rho(it, seed + i)))
        return out
    if kind == "gf":
        return _exact_gf(case, seed)
    if kind == "ts":
        return _exact_ts(case, seed)
    return _exact_net(case, seed)
