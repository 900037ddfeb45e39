"""Timed cases of the public entry points: PSATD steps (Plan, Batch, Local), FDTD steps
and the far-field transform, over the sizes, precisions, source forms and schemes that
the repository's workloads use.

Every case is ONE call of a user's program: a particle-in-cell loop deposits new currents
before each field step, so a grid's case is one step (``nsteps`` = 1); the batched and
the 2D FDTD cases advance several steps per call, as runs with a held source do.  Fields
are advanced in place, and the returned arrays are the state's own.
"""
from __future__ import annotations

import math

import torch

from paper_1608_05739_gb300 import capi, synth

DEV = "cuda"
SQ2 = math.sqrt(0.5)
PRESENT = capi.PRESENT  # layout -> components present in (E, B, J)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the accuracy workload: 2D vacuum, all components, FP64 (the smallest grid in use)
        dict(name="vac128_fp64", kind="plan", nx=128, ny=128, nz=0, layout="2d6", prec="fp64", src="none", order=0),
        # a small local domain with sides 3 * 2^k and 5 * 2^k: latency and launches count
        dict(name="te192x80_fp32", kind="plan", nx=192, ny=80, nz=0, layout="te", prec="fp32", src="J", order=0),
        # the plasma-mirror grid: 2D TE, one step per deposited current
        dict(name="te2048_fp32", kind="plan", nx=2048, ny=2048, nz=0, layout="te", prec="fp32", src="J", order=0),
        # 3D charges with the rho-form
        dict(name="rho256_fp32", kind="plan", nx=256, ny=256, nz=256, layout="3d6", prec="fp32", src="rho", order=0),
        # the large 3D grid (11.8 GB of fields and sources)
        dict(name="rho512x512x1024_fp32", kind="plan", nx=512, ny=512, nz=1024, layout="3d6", prec="fp32", src="rho",
             order=0),
        # the tensor-core path in 3D (split FP16)
        dict(name="j256_fp16", kind="plan", nx=256, ny=256, nz=256, layout="3d6", prec="mixed_fp16", src="J", order=0),
        # the batched local domains: 512 patches, split BF16 on power-of-two sides, and FP32 on its own sides
        dict(name="batch512_bf16", kind="batch", npatch=512, prec="mixed_bf16", layout="te", src="J", nsteps=4),
        dict(name="batch512_fp32", kind="batch", npatch=512, prec="fp32", layout="te", src="J", nsteps=4),
        # local FFTs with guard cells at the order they are meant for
        dict(name="local3840_order16", kind="local", ix=240, iy=240, px=16, py=8, guard=8, layout="te", prec="fp32",
             src="J", order=16),
        # the FDTD comparators: Yee in 3D (one step per call), CKC in 2D (several steps of a held source)
        dict(name="yee256_fp32", kind="fdtd", nx=256, ny=256, nz=256, scheme="yee", layout="3d6", prec="fp32", src="J",
             nsteps=1),
        dict(name="ckc2048_fp32", kind="fdtd", nx=2048, ny=2048, nz=0, scheme="ckc", layout="te", prec="fp32", src="J",
             nsteps=8),
        # the harmonic diagnostic: 8 harmonics x 481 directions over the reflected window of a snapshot
        dict(name="farfield_8x481", kind="farfield", nx=4096, ny=1024, x0=512, wx=512, wy=1024, nk=8 * 481,
             window="x", prec="fp32"),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _length(rng, lo, hi, prec, half=False):
    """A transform length in [lo, hi]: 2^k, and in FP32 also 3 * 2^k and 5 * 2^k (``half``: of nx/2)."""
    cand = [1 << k for k in range(3, 13)]
    if prec == "fp32":
        cand += [3 << k for k in range(4, 11)] + [5 << k for k in range(4, 9)]
    cand = [2 * v if half else v for v in cand]
    cand = sorted(v for v in cand if lo <= v <= hi)
    target = _loguniform(rng, lo, hi)
    return min(cand, key=lambda v: abs(math.log(v / target)))


def draw(rng):
    kind = rng.choice(["plan2", "plan2", "plan3", "batch", "local", "fdtd2", "fdtd3", "farfield"])
    if kind == "plan2":
        layout = rng.choice(["te", "te", "tm", "2d6"])
        prec = rng.choice(["fp32", "fp32", "fp64", "mixed_fp16", "mixed_bf16"])
        src = rng.choice(["none", "J", "J"] if layout == "tm" else ["none", "J", "J", "rho"])
        lo, hi = (256, 2048) if prec.startswith("mixed") else (64, 1024) if prec == "fp64" else (64, 2048)
        return dict(kind="plan", nx=_length(rng, lo, hi, prec, True), ny=_length(rng, lo, hi, prec), nz=0,
                    layout=layout, prec=prec, src=src, order=rng.choice([0, 0, 8, 16]))
    if kind == "plan3":
        prec = rng.choice(["fp32", "fp32", "fp32", "mixed_fp16"])
        lo = 128 if prec == "mixed_fp16" else 48
        return dict(kind="plan", nx=_length(rng, max(lo, 96), 512, prec, True), ny=_length(rng, lo, 512, prec),
                    nz=_length(rng, lo, 512, prec), layout="3d6", prec=prec, src=rng.choice(["none", "J", "rho"]),
                    order=rng.choice([0, 0, 128]))
    if kind == "batch":
        return dict(kind="batch", npatch=int(_loguniform(rng, 8, 512)), prec=rng.choice(["fp32", "mixed_bf16"]),
                    layout="te", src="J", nsteps=rng.choice([1, 2, 3, 4]))
    if kind == "local":
        g = rng.randrange(8, 17)
        ex, ey = rng.choice([96, 128, 192, 256]), rng.choice([96, 128, 192, 256])
        return dict(kind="local", ix=ex - 2 * g, iy=ey - 2 * g, px=rng.randrange(2, 13), py=rng.randrange(2, 13),
                    guard=g, layout="te", prec="fp32", src=rng.choice(["none", "J"]), order=rng.choice([8, 16]))
    if kind == "fdtd2":
        layout = rng.choice(["te", "tm", "2d6"])
        return dict(kind="fdtd", nx=int(_loguniform(rng, 64, 2048)), ny=int(_loguniform(rng, 64, 2048)), nz=0,
                    scheme=rng.choice(["yee", "ckc"]), layout=layout, prec=rng.choice(["fp32", "fp32", "fp64"]),
                    src=rng.choice(["none", "J"]), nsteps=rng.randrange(1, 9))
    if kind == "fdtd3":
        return dict(kind="fdtd", nx=int(_loguniform(rng, 32, 384)), ny=int(_loguniform(rng, 32, 256)),
                    nz=int(_loguniform(rng, 32, 256)), scheme="yee", layout="3d6", prec="fp32",
                    src=rng.choice(["none", "J"]), nsteps=rng.randrange(1, 4))
    wx, wy = int(_loguniform(rng, 64, 1024)), int(_loguniform(rng, 64, 1024))
    x0 = rng.randrange(0, 512)
    return dict(kind="farfield", nx=x0 + wx + rng.randrange(0, 512), ny=wy + rng.randrange(0, 64), x0=x0, wx=wx, wy=wy,
                nk=int(_loguniform(rng, 16, 4096)), window=rng.choice(["none", "x", "xy"]),
                prec=rng.choice(["fp32", "fp32", "fp64"]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _k2(shape):
    """Squared wavenumbers of the half spectrum (unit cells), broadcast over the axes."""
    nd, out = len(shape), None
    for ax, n in enumerate(shape):
        f = (torch.fft.rfftfreq if ax == nd - 1 else torch.fft.fftfreq)(n, device=DEV) * (2 * math.pi)
        f = (f * f).view([-1 if i == ax else 1 for i in range(nd)])
        out = f if out is None else out + f
    return out


def _field(gen, shape, dtype):
    """A random field of unit rms with spectral power ~ |k|^-2."""
    k2 = _k2(shape)
    F = torch.fft.rfftn(torch.randn(shape, device=DEV, generator=gen))
    F *= torch.rsqrt(torch.clamp(k2, min=(2 * math.pi / max(shape)) ** 2))
    f = torch.fft.irfftn(F, s=shape)
    return (f / f.square().mean().sqrt()).to(dtype)


def _source(gen, shape, dtype, scale=0.01):
    """Noise smoothed to a Gaussian of three cells (macro-charges): current and charge densities."""
    F = torch.fft.rfftn(torch.randn(shape, device=DEV, generator=gen)) * torch.exp(-4.5 * _k2(shape))
    f = torch.fft.irfftn(F, s=shape)
    return (f * (scale / f.square().mean().sqrt())).to(dtype)


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _grid_inputs(case, seed, shape, make_field, make_source):
    g, dt = _gen(seed), _dtype(case)
    pe, pb, pj = PRESENT[case["layout"]]
    E = [make_field(g, shape, dt) if p else None for p in pe]
    B = [make_field(g, shape, dt) if p else None for p in pb]
    J = [make_source(g, shape, dt) if p and case["src"] != "none" else None for p in pj]
    rho = [None, None]
    if case["src"] == "rho":
        rho[0] = make_source(g, shape, dt)
        rho[1] = rho[0] + 0.1 * make_source(g, shape, dt)  # the charges moved by a fraction of a cell
    return dict(E=E, B=B, J=J if case["src"] != "none" else None, rho=rho)


def _shape(case):
    if case["kind"] == "local":
        return (case["py"] * case["iy"], case["px"] * case["ix"])
    return (case["nz"], case["ny"], case["nx"]) if case["nz"] else (case["ny"], case["nx"])


def _patches(case):
    sizes, _ = synth.batch_patch_sizes(case["npatch"], 1612, mixed_ok=case["prec"] == "fp32")
    return sizes


def _white(scale):
    return lambda g, shape, dt: torch.randn(shape, device=DEV, generator=g).mul_(scale).to(dt)


def _inputs(case, seed):
    if case["kind"] == "batch":
        n = sum(a * b for a, b in _patches(case))
        return _grid_inputs(case, seed, (n,), _white(0.1), _white(0.01))
    if case["kind"] == "farfield":
        g = _gen(seed)
        F = _field(g, (case["ny"], case["nx"]), _dtype(case))
        # rings |k| = n k0 of the harmonics n = 1..8 of a wave of 64 cells, directions over +-80 degrees
        j = torch.arange(case["nk"], device=DEV, dtype=torch.float64)
        per = max(1, case["nk"] // 8)
        k = (2 * math.pi / 64.0) * (1 + torch.clamp(torch.div(j, per, rounding_mode="floor"), max=7))
        th = (torch.rand(case["nk"], device=DEV, generator=g, dtype=torch.float64) - 0.5) * (160.0 / 180.0 * math.pi)
        return dict(F=F, k=torch.stack([k * torch.cos(th), k * torch.sin(th)], dim=1).contiguous())
    return _grid_inputs(case, seed, _shape(case), _field, _source)


def _dt(case):
    """c dt in cells: the Courant-free PSATD grids run at 1/sqrt(2) (the FP64 one at 1/2), FDTD inside its limit."""
    if case["kind"] == "fdtd":
        return 0.5
    return 0.5 if case["prec"] == "fp64" else SQ2


# ------------------------------------------------------------------ entry points
def prepare(case, seed):
    st = _inputs(case, seed)
    st["case"] = case
    kind, opts = case["kind"], dict(layout=case.get("layout"), prec=case["prec"], src=case.get("src"))
    if kind == "plan":
        n = (case["nx"], case["ny"], case["nz"]) if case["nz"] else (case["nx"], case["ny"])
        st["solver"] = capi.Plan(n, (1.0,) * len(n), _dt(case), order=case["order"], **opts)
    elif kind == "local":
        ny, nx = _shape(case)
        st["solver"] = capi.Local((nx, ny), (1.0, 1.0), _dt(case), px=case["px"], py=case["py"], guard=case["guard"],
                                  order=case["order"], **opts)
    elif kind == "batch":
        # multi-step calls replay a recorded graph, which needs a stream of their own
        st["stream"] = torch.cuda.Stream()
        st["solver"] = capi.Batch(_patches(case), (1.0, 1.0), _dt(case), stream=st["stream"], **opts)
    return st


def _fields_out(st):
    return [f for f in st["E"] + st["B"] if f is not None]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "farfield":
        return capi.farfield((case["nx"], case["ny"]), (1.0, 1.0), st["F"], st["k"],
                             x_range=(case["x0"], case["x0"] + case["wx"]), y_range=(0, case["wy"]),
                             window=case["window"])
    if kind == "fdtd":
        n = (case["nx"], case["ny"], case["nz"]) if case["nz"] else (case["nx"], case["ny"])
        capi.fdtd_step(n, (1.0,) * len(n), _dt(case), st["E"], st["B"], st["J"], scheme=case["scheme"],
                       layout=case["layout"], prec=case["prec"], nsteps=case["nsteps"])
    elif kind == "batch":
        cur = torch.cuda.current_stream()
        st["stream"].wait_stream(cur)
        st["solver"].step(st["E"], st["B"], st["J"], nsteps=case["nsteps"])
        cur.wait_stream(st["stream"])
    else:
        st["solver"].step(st["E"], st["B"], st["J"], st["rho"][0], st["rho"][1])
    return _fields_out(st)


# ------------------------------------------------------------------ work and tolerances
def work(case):
    es = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "farfield":
        cells = case["wx"] * case["wy"]
        return dict(bytes=cells * es + case["nk"] * 32.0, flops=4.0 * cells * case["nk"])
    pe, pb, pj = PRESENT[case["layout"]]
    nf = sum(pe) + sum(pb)
    ns = 0 if case["src"] == "none" else sum(pj) + (2 if case["src"] == "rho" else 0)
    steps = case.get("nsteps", 1)
    if case["kind"] == "fdtd":  # per step: fields read and written, sources read
        cells = math.prod(_shape(case))
        return dict(bytes=float(steps * cells * es * (2 * nf + ns)), flops=float(steps * cells * nf * 12))
    if case["kind"] == "batch":
        grids = _patches(case)
    elif case["kind"] == "local":
        grids = [(case["ix"] + 2 * case["guard"], case["iy"] + 2 * case["guard"])] * (case["px"] * case["py"])
    else:
        grids = [tuple(reversed(_shape(case)))]
    cells = sum(math.prod(g) for g in grids)
    moved = math.prod(_shape(case)) if case["kind"] == "local" else cells
    # real transforms (2.5 N log2 N each) and about 12 operations per component and mode (N/2 of them)
    fl = sum(math.prod(g) * (2.5 * math.log2(math.prod(g)) * (2 * nf + ns) + 6 * (2 * nf + ns)) for g in grids)
    return dict(bytes=float(steps * moved * es * (2 * nf + ns)), flops=float(steps * fl))


def tolerance(case):
    """About four times the error of one call against `exact` (rel: of each output in the 2-norm; max: largest
    difference over the rms): PSATD 4.8e-16 in FP64, 1.5e-7 .. 4.1e-7 in FP32 and the mixed precisions, FDTD 1.6e-7,
    the far field 3.7e-8 (rows summed in FP32) and 3.0e-16."""
    if case["prec"] == "fp64":
        return dict(rel=2e-15, max=2e-14)
    if case["kind"] == "farfield":
        return dict(rel=1.5e-7, max=2e-6)
    if case["kind"] == "fdtd":
        return dict(rel=6e-7, max=4e-6)
    return dict(rel=1.6e-6, max=1e-5)


# ------------------------------------------------------------------ the same in 64 bits, plain torch
def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _weights(p):
    """Staggered first-derivative weights of order p: C_l solves sum_l C_l (2l-1)^(2m-1) = delta_m1."""
    h, out = p // 2, []
    for ell in range(1, h + 1):
        v = 1.0 / (2 * ell - 1)
        for m in range(1, h + 1):
            if m != ell:
                v *= (2 * m - 1) ** 2 / ((2 * m - 1) ** 2 - (2 * ell - 1) ** 2)
        out.append(v)
    return out


class _Exact:
    """PSATD on periodic grids of ``shape`` (unit cells; the leading axis may batch grids of one size)."""

    def __init__(self, shape, dt, order):
        nd = len(shape)
        self.shape, self.dims, self.dt, self.order = shape, tuple(range(-nd, 0)), dt, order
        raw = []
        for ax in range(nd - 1, -1, -1):
            n = shape[ax]
            f = (torch.fft.rfftfreq if ax == nd - 1 else torch.fft.fftfreq)(n, device=DEV, dtype=torch.float64)
            raw.append((2 * math.pi * f).view([-1 if i == ax else 1 for i in range(nd)]))
        zero = torch.zeros([1] * nd, device=DEV, dtype=torch.float64)
        raw += [zero] * (3 - nd)
        if order:
            ws = _weights(order)
            self.k = [2 * sum(w * torch.sin((2 * i + 1) * 0.5 * k) for i, w in enumerate(ws)) for k in raw]
            self.ph = [torch.exp(-0.5j * k) for k in raw]
        else:
            self.k = [torch.where((k.abs() - math.pi).abs() < 1e-9, torch.zeros_like(k), k) for k in raw]
        kx, ky, kz = self.k
        self.k2 = kx * kx + ky * ky + kz * kz
        x = self.x = torch.sqrt(self.k2) * dt
        self.C, self.sinc = torch.cos(x), torch.sinc(x / math.pi)
        self.h2 = 0.5 * torch.sinc(0.5 * x / math.pi) ** 2  # (1 - C) / x^2
        xs, x2 = torch.where(x < 0.5, torch.ones_like(x), x), x * x
        s1, s2 = torch.zeros_like(x), torch.zeros_like(x)
        for n in range(11, 0, -1):
            s1 = s1 * x2 + (-1) ** n / math.factorial(2 * n + 1)
            s2 = s2 * x2 + (-1) ** (n + 1) * 2 * n / math.factorial(2 * n + 1)
        self.f1 = torch.where(x < 0.5, s1, (torch.sin(xs) / xs - 1) / xs ** 2)            # (sinc - 1) / x^2
        self.f2 = torch.where(x < 0.5, s2, (torch.sin(xs) / xs - torch.cos(xs)) / xs ** 2)  # (sinc - C) / x^2

    SE, SB = ((0,), (1,), (2,)), ((1, 2), (0, 2), (0, 1))

    def fwd(self, f, axes):
        if f is None:
            return 0.0
        F = torch.fft.rfftn(f.double(), dim=self.dims)
        for a in axes if self.order else ():
            F = F * self.ph[a]
        return F

    def inv(self, F, axes):
        for a in axes if self.order else ():
            F = F * self.ph[a].conj()
        return torch.fft.irfftn(F, s=self.shape, dim=self.dims)

    def step(self, E, B, J, rho, form):
        """One step; E, B, J, rho real arrays (None: absent), the new E, B (None where absent)."""
        k, dt = self.k, self.dt
        Eh = [self.fwd(E[i], self.SE[i]) for i in range(3)]
        Bh = [self.fwd(B[i], self.SB[i]) for i in range(3)]
        Jh = [self.fwd(J[i], self.SE[i]) for i in range(3)] if form != "none" else [0.0] * 3
        along = sum(k[i] * Bh[i] for i in range(3)) * (dt * dt * self.h2)
        kE, kJ = _cross(k, Eh), _cross(k, Jh)
        Bn = [self.inv(self.C * Bh[i] + k[i] * along - 1j * dt * self.sinc * kE[i] + 1j * dt * dt * self.h2 * kJ[i],
                       self.SB[i]) if B[i] is not None else None for i in range(3)]
        del along, kE, kJ
        kB = _cross(k, Bh)
        del Bh
        if form == "rho":
            pot = 1j * dt * dt * (self.f1 * self.fwd(rho[1], ()) - self.f2 * self.fwd(rho[0], ()))
        else:
            pot = sum(k[i] * Eh[i] for i in range(3)) * (dt * dt * self.h2)
            if form == "J":
                pot = pot + sum(k[i] * Jh[i] for i in range(3)) * (dt ** 3 * self.f1)
        En = [self.inv(self.C * Eh[i] + 1j * dt * self.sinc * kB[i] - dt * self.sinc * Jh[i] + k[i] * pot,
                       self.SE[i]) if E[i] is not None else None for i in range(3)]
        return En, Bn


def _none(v, f):
    return [None if x is None else f(x) for x in v]


def _exact_psatd(case, s):
    ex = _Exact(_shape(case), _dt(case), case["order"])
    En, Bn = ex.step(s["E"], s["B"], s["J"], s["rho"], case["src"])
    return [f for f in En + Bn if f is not None]


def _exact_batch(case, s):
    sizes = _patches(case)
    off, acc = [], 0
    for a, b in sizes:
        off.append(acc)
        acc += a * b
    out = [torch.empty(acc, dtype=torch.float64, device=DEV) for f in s["E"] + s["B"] if f is not None]
    for nx, ny in sorted(set(sizes)):
        idx = [i for i, ab in enumerate(sizes) if ab == (nx, ny)]
        ex = _Exact((ny, nx), _dt(case), 0)
        for c0 in range(0, len(idx), 32):
            part = idx[c0:c0 + 32]

            def take(f):
                return torch.stack([f[off[i]:off[i] + nx * ny].view(ny, nx) for i in part]).double()

            E, B, J = _none(s["E"], take), _none(s["B"], take), _none(s["J"], take)
            for _ in range(case["nsteps"]):
                E, B = ex.step(E, B, J, None, case["src"])
            for o, f in zip(out, [f for f in E + B if f is not None]):
                for j, i in enumerate(part):
                    o[off[i]:off[i] + nx * ny] = f[j].reshape(-1)
    return out


def _exact_local(case, s):
    ix, iy, px, py, g = (case[v] for v in ("ix", "iy", "px", "py", "guard"))
    ny, nx = _shape(case)
    yi = (torch.arange(py, device=DEV)[:, None] * iy - g + torch.arange(iy + 2 * g, device=DEV)[None, :]) % ny
    xi = (torch.arange(px, device=DEV)[:, None] * ix - g + torch.arange(ix + 2 * g, device=DEV)[None, :]) % nx

    def take(f):  # [py, px, ey, ex]
        return f.double()[yi][:, :, xi].permute(0, 2, 1, 3)

    def put(f):
        return f[:, :, g:g + iy, g:g + ix].permute(0, 2, 1, 3).reshape(ny, nx)

    ex = _Exact((iy + 2 * g, ix + 2 * g), _dt(case), case["order"])
    J = _none(s["J"], take) if s["J"] is not None else None
    En, Bn = ex.step(_none(s["E"], take), _none(s["B"], take), J, None, case["src"])
    return [put(f) for f in En + Bn if f is not None]


def _exact_fdtd(case, s):
    """B half step, E step, B half step; forward differences of E, backward of B (x is the last axis)."""
    E, B = _none(s["E"], lambda f: f.double()), _none(s["B"], lambda f: f.double())
    J = _none(s["J"], lambda f: f.double()) if s["J"] is not None else [None] * 3
    three, ckc, dt = case["nz"] > 0, case["scheme"] == "ckc", _dt(case)

    def diff(f, a, fw):
        if f is None or (a == 2 and not three):
            return 0.0
        d = torch.roll(f, -1, -1 - a) - f if fw else f - torch.roll(f, 1, -1 - a)
        if fw and ckc:
            t = -2 + a  # the transverse axis
            d = 0.75 * d + 0.125 * (torch.roll(d, 1, t) + torch.roll(d, -1, t))
        return d

    def curl(F, i, fw):
        i1, i2 = (i + 1) % 3, (i + 2) % 3
        return diff(F[i2], i1, fw) - diff(F[i1], i2, fw)

    def faraday(B):
        return [None if B[i] is None else B[i] - 0.5 * dt * curl(E, i, True) for i in range(3)]

    for _ in range(case["nsteps"]):
        B = faraday(B)
        E = [None if E[i] is None else E[i] + dt * curl(B, i, False) - (dt * J[i] if J[i] is not None else 0.0)
             for i in range(3)]
        B = faraday(B)
    return [f for f in E + B if f is not None]


def _exact_farfield(case, s):
    x0, wx, wy = case["x0"], case["wx"], case["wy"]
    F = s["F"][:wy, x0:x0 + wx].double()

    def hann(n, on):
        i = torch.arange(n, device=DEV, dtype=torch.float64)
        return torch.sin(math.pi * (i + 0.5) / n) ** 2 if on else torch.ones_like(i)

    x = torch.arange(x0, x0 + wx, device=DEV, dtype=torch.float64)
    y = torch.arange(wy, device=DEV, dtype=torch.float64)
    out = []
    for k in s["k"].split(256):
        ax = torch.exp(-1j * k[:, :1] * x) * hann(wx, case["window"] != "none")
        ay = torch.exp(-1j * k[:, 1:] * y) * hann(wy, case["window"] == "xy")
        rows = torch.complex(ax.real @ F.T, ax.imag @ F.T)  # [k, wy]
        out.append((rows * ay).sum(1))
    return torch.cat(out)


def exact(case, seed):
    s = _inputs(case, seed)
    kind = {"plan": _exact_psatd, "batch": _exact_batch, "local": _exact_local, "fdtd": _exact_fdtd,
            "farfield": _exact_farfield}[case["kind"]]
    return kind(case, s)
