"""Performance cases of the field advance: what its users have it do, each
through the public entry points (``fmx.Grid``, the ``fmx_batch_*`` calls, the
autograd function of ``adjoint.py``).

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from
the seed alone, ``run`` makes one pass, ``exact`` evaluates the same pass in
FP64 with plain torch operations (whole-array periodic shifts, in the notation
of ``include/fmx.h``, on the coefficients rounded to the grid's precision as
``fmx_coefficients`` documents them), and ``work`` counts the bytes and
floating-point operations the pass cannot do without.

Kinds: ``advance`` (a time loop between two looks at the fields), ``coupled``
(a particle code's loop: every step brings its own current), ``residual``
(Algorithm 1 to a residual target), ``monitor`` (advance, post-process filter,
energy and divergence diagnostics), ``batch`` (many independent grids) and
``gradient`` (forward run and its adjoint).
"""
import ctypes
import math

import numpy as np
import torch

from paper_1907_13088_gb300 import fmx
from paper_1907_13088_gb300.adjoint import GaussSourceRun, make_function

DEV = "cuda" if torch.cuda.is_available() else "cpu"
AX = (-1, -2, -3)  # array axis of x, y, z


def listed():
    return [
        # the smallest call: one step of a small 2D grid inside a particle
        # loop, which hands over the current it has just deposited
        dict(name="coupled 64x64 f32", kind="coupled", nx=64, ny=64, nz=1, f64=False, m=4, passes=1, steps=1),
        # an ordinary 2D run of a few thousand cells per SM
        dict(name="advance 512x512 f32", kind="advance", nx=512, ny=512, nz=1, f64=False, m=4, passes=3, current=True,
             steps=4),
        # the benchmark's 2D grid: four sweeps, three filter passes
        dict(name="advance 4096x4096 f32", kind="advance", nx=4096, ny=4096, nz=1, f64=False, m=4, passes=3,
             current=True, steps=4),
        # sizes a user picks from the physics, odd on both axes
        dict(name="advance 1537x1023 f32", kind="advance", nx=1537, ny=1023, nz=1, f64=False, m=3, passes=2,
             current=True, steps=4),
        # a double-precision 2D run (convergence and dispersion studies)
        dict(name="advance 2048x1536 f64", kind="advance", nx=2048, ny=1536, nz=1, f64=True, m=4, passes=3,
             current=True, steps=1),
        # the benchmark's 3D grid, the largest case
        dict(name="advance 512^3 f32", kind="advance", nx=512, ny=512, nz=512, f64=False, m=4, passes=1, current=True,
             steps=1),
        # a ragged 3D box with an odd row length
        dict(name="advance 201x150x99 f32", kind="advance", nx=201, ny=150, nz=99, f64=False, m=4, passes=1,
             current=True, steps=2),
        # 3D in double precision
        dict(name="advance 128x128x96 f64", kind="advance", nx=128, ny=128, nz=96, f64=True, m=4, passes=1,
             current=True, steps=1),
        # the 64 x 64 plane-wave study: every step solved to 1e-13
        dict(name="residual 64x64 f64", kind="residual", nx=64, ny=64, nz=1, f64=True, tol=1e-13, steps=20),
        # a monitored run: steps, one post-process pass, energies and divergences
        dict(name="monitor 1536x1200 f32", kind="monitor", nx=1536, ny=1200, nz=1, f64=False, m=4, passes=1, steps=4),
        # the batch of 256 uneven grids with their own Courant numbers
        dict(name="batch 256 grids f32", kind="batch", count=256, lo=64, hi=1024, m=4, sizes_seed=1907004, steps=4),
        # the differentiable Gaussian-source run: forward, loss, adjoint
        dict(name="gradient 1024x1024 f32", kind="gradient", nx=1024, ny=1024, m=4, passes=3, sources=64, steps=10,
             every=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges (any parity of the sizes)."""
    kind = rng.choice(["coupled", "advance2", "advance2", "advance2d64", "advance3", "advance3", "advance3d64",
                       "residual", "monitor", "batch", "gradient"])
    if kind == "coupled":
        return dict(kind="coupled", nx=_log(rng, 32, 384), ny=_log(rng, 32, 384), nz=1, f64=False,
                    m=rng.randint(2, 4), passes=rng.randint(0, 3), steps=1)
    if kind == "advance2":
        return dict(kind="advance", nx=_log(rng, 64, 4096), ny=_log(rng, 64, 4096), nz=1, f64=False,
                    m=rng.randint(1, 4), passes=rng.randint(0, 3), current=rng.random() < 0.75,
                    steps=rng.randint(1, 8))
    if kind == "advance2d64":
        return dict(kind="advance", nx=_log(rng, 64, 2048), ny=_log(rng, 64, 2048), nz=1, f64=True,
                    m=rng.randint(2, 4), passes=rng.randint(0, 3), current=rng.random() < 0.75,
                    steps=rng.randint(1, 2))
    if kind == "advance3":
        return dict(kind="advance", nx=_log(rng, 32, 400), ny=_log(rng, 32, 400), nz=_log(rng, 32, 400), f64=False,
                    m=rng.randint(2, 4), passes=rng.randint(0, 1), current=rng.random() < 0.75, steps=1)
    if kind == "advance3d64":
        return dict(kind="advance", nx=_log(rng, 24, 160), ny=_log(rng, 24, 160), nz=_log(rng, 24, 160), f64=True,
                    m=rng.randint(2, 4), passes=rng.randint(0, 1), current=rng.random() < 0.75, steps=1)
    if kind == "residual":
        f64 = rng.random() < 0.5
        return dict(kind="residual", nx=_log(rng, 32, 320), ny=_log(rng, 32, 320), nz=1, f64=f64,
                    tol=1e-13 if f64 else 1e-5, steps=rng.randint(2, 20))
    if kind == "monitor":
        two = rng.random() < 0.5
        return dict(kind="monitor", nx=_log(rng, 64, 1536 if two else 160), ny=_log(rng, 64, 1536 if two else 160),
                    nz=1 if two else _log(rng, 32, 128), f64=rng.random() < 0.25, m=rng.randint(2, 4),
                    passes=rng.randint(1, 2), steps=rng.randint(1, 6))
    if kind == "batch":
        return dict(kind="batch", count=_log(rng, 16, 256), lo=64, hi=_log(rng, 128, 1024), m=rng.choice([2, 4]),
                    sizes_seed=rng.randint(1, 10**6), steps=2 * rng.randint(1, 3))
    return dict(kind="gradient", nx=_log(rng, 96, 1200), ny=_log(rng, 96, 1200), m=rng.randint(2, 4),
                passes=rng.randint(0, 3), sources=rng.randint(1, 96), steps=rng.randint(4, 12),
                every=rng.randint(2, 6))


# ---------------------------------------------------------------------------
# inputs


def _shape(case):
    nz = case.get("nz", 1)
    return (case["nx"], case["ny"], nz) if nz > 1 else (case["nx"], case["ny"])


def _spectrum(shape, gen, weight, dtype):
    """Real field with the given mode amplitudes and random phases, unit RMS."""
    f = torch.fft.irfftn(torch.polar(weight, 2 * math.pi * torch.rand(weight.shape, generator=gen, device=DEV)),
                         s=shape)
    return (f / f.square().mean().sqrt()).to(dtype)


def _modes(shape):
    n = torch.zeros((), device=DEV)
    for a, s in enumerate(shape):
        q = torch.fft.rfftfreq(s, 1.0 / s, device=DEV) if a == len(shape) - 1 else torch.fft.fftfreq(s, 1.0 / s, device=DEV)
        n = n + q.square().reshape([-1 if b == a else 1 for b in range(len(shape))])
    return n.sqrt()


def _curl(p, sign):
    """Staggered curl of a potential: backward (sign 1) or forward (-1) differences."""
    def d(f, ax):
        return sign * (f - torch.roll(f, sign, ax)) if f.shape[ax] > 1 else torch.zeros_like(f)
    return torch.stack([d(p[2], -2) - d(p[1], -3), d(p[0], -3) - d(p[2], -1), d(p[1], -1) - d(p[0], -2)])


def _fields(nx, ny, nz, seed, dtype, width=16.0):
    """Divergence-free E and B whose power falls as |n|^-2 up to n = N/8, unit
    RMS, and the solenoidal current of a smooth random potential."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    shape = (nz, ny, nx)
    n = _modes(shape)
    kmax = max(2.0, max(shape) / 8)
    w = torch.where((n >= 1) & (n <= kmax), n.clamp(min=1.0) ** -2, torch.zeros_like(n))
    out = []
    for sign in (1, -1):
        F = _curl([_spectrum(shape, gen, w, torch.float32) for _ in range(3)], sign)
        out.append((F / F.square().mean().sqrt()).to(dtype))
    k2 = torch.zeros((), device=DEV)
    for a, s in enumerate(shape):
        q = torch.fft.rfftfreq(s, device=DEV) if a == 2 else torch.fft.fftfreq(s, device=DEV)
        k2 = k2 + (2 * math.pi * q).square().reshape([-1 if b == a else 1 for b in range(3)])
    wj = torch.exp(-0.5 * k2 * width * width)
    wj[0, 0, 0] = 0.0
    if float(wj.sum()) == 0.0:  # a box too small for the width: its lowest modes
        wj[..., 1] = 1.0
    J = _curl([_spectrum(shape, gen, wj, torch.float32) for _ in range(3)], 1)
    J = (1e-3 * J / J.square().mean().sqrt()).to(dtype)
    return out[0], out[1], J


def _raw_fields(nx, ny, nz, seed, dtype):
    """E and B interpolated from elsewhere: the same spectrum, but with a charge
    density and a divergence of B for the monitor to report."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    shape = (nz, ny, nx)
    n = _modes(shape)
    w = torch.where((n >= 1) & (n <= max(2.0, max(shape) / 8)), n.clamp(min=1.0) ** -1, torch.zeros_like(n))
    F = torch.stack([_spectrum(shape, gen, w, torch.float32) for _ in range(6)]).to(dtype)
    return F[:3], F[3:]


def _plane_waves(nx, ny, seed, dt, dtype):
    """Eight vacuum plane waves (E_z, B_x, B_y), integer modes up to |n| = 8."""
    rng = np.random.default_rng(seed)
    cand = [(a, b) for a in range(-8, 9) for b in range(-8, 9) if 1 <= a * a + b * b <= 64 and (a > 0 or (a == 0 and b > 0))]
    x = torch.arange(nx, device=DEV, dtype=torch.float64)[None, :]
    y = torch.arange(ny, device=DEV, dtype=torch.float64)[:, None]
    E = torch.zeros((3, 1, ny, nx), device=DEV, dtype=torch.float64)
    B = torch.zeros_like(E)
    for i in rng.choice(len(cand), size=8, replace=False):
        kx, ky = 2 * math.pi * cand[i][0] / nx, 2 * math.pi * cand[i][1] / ny
        k, amp, ph = math.hypot(kx, ky), rng.standard_normal(), rng.uniform(0, 2 * math.pi)
        E[2, 0] += amp * torch.cos(kx * x + ky * y + ph)
        B[0, 0] += ky / k * amp * torch.cos(kx * x + ky * (y + 0.5) - 0.5 * k * dt + ph)
        B[1, 0] -= kx / k * amp * torch.cos(kx * (x + 0.5) + ky * y - 0.5 * k * dt + ph)
    return E.to(dtype), B.to(dtype)


def _dt(shape, courant):
    return courant / math.sqrt(len(shape))  # unit cells, c = 1


def _dtype(case):
    return torch.float64 if case.get("f64") else torch.float32


def _inputs(case, seed):
    nx, ny, nz, dt = case["nx"], case["ny"], case.get("nz", 1), _dtype(case)
    if case["kind"] == "residual":
        E, B = _plane_waves(nx, ny, seed, _dt(_shape(case), 0.5), dt)
        return E, B, None
    if case["kind"] == "monitor":
        E, B = _raw_fields(nx, ny, nz, seed, dt)
        return E, B, None
    E, B, J = _fields(nx, ny, nz, seed, dt)
    return E, B, J if case["kind"] == "coupled" or case.get("current") else None


def _batch_sizes(case):
    rng = np.random.default_rng(case["sizes_seed"])
    draws = lambda: np.round(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["count"]))).astype(int)
    nx, ny = draws(), draws()
    cf = rng.uniform(0.3, 0.9, case["count"])
    return [(int(a), int(b), float(c)) for a, b, c in zip(nx, ny, cf)]


def _batch_layout(case):
    """Per grid: sizes, Courant number, pitch, offset of its first component,
    elements per component; and the elements of a whole state set."""
    rows, off = [], 0
    for nx, ny, cf in _batch_sizes(case):
        pitch = (nx + 3) // 4 * 4
        size = (pitch * ny + 63) // 64 * 64
        rows.append((nx, ny, cf, pitch, off, size))
        off += 6 * size
    return rows, off


def _batch_fields(case, seed):
    """Every grid's E and B in one array, in the layout of _batch_layout."""
    rows, total = _batch_layout(case)
    slab = torch.zeros(total, dtype=torch.float32, device=DEV)
    for i, (nx, ny, _, pitch, off, size) in enumerate(rows):
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed * 1000 + i)
        n = _modes((ny, nx))
        w = torch.where((n >= 1) & (n <= max(nx, ny) / 8), n.clamp(min=1.0) ** -1, torch.zeros_like(n))
        F = torch.fft.irfftn(torch.polar(w.expand(6, -1, -1), 2 * math.pi * torch.rand((6,) + w.shape, generator=gen, device=DEV)),
                             s=(ny, nx), dim=(1, 2))
        F = F / F.square().mean().sqrt()
        for c in range(6):
            slab[off + c * size:off + c * size + pitch * ny].view(ny, pitch)[:, :nx] = F[c]
    return slab


def _gradient_inputs(case, seed):
    rng = np.random.default_rng(seed)
    nx, ny, n = case["nx"], case["ny"], case["sources"]
    cxy = np.stack([rng.uniform(0, nx, n), rng.uniform(0, ny, n)], axis=1)
    phases, theta = rng.uniform(0.0, 2.0 * math.pi, n), rng.standard_normal(n)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    F = 0.01 * torch.randn((6, ny, nx), generator=gen, device=DEV)
    win = torch.zeros((1, ny, nx), device=DEV)
    win[:, 7 * ny // 16:9 * ny // 16, 7 * nx // 16:9 * nx // 16] = 1.0
    return cxy, phases, theta, F[:3].contiguous(), F[3:].contiguous(), win


# ---------------------------------------------------------------------------
# the passes


class _BatchState:
    """A batch on buffers of the caller's own, through the batch entry points."""

    def __init__(self, case, seed):
        rows, total = _batch_layout(case)
        self.stream = torch.cuda.Stream()
        self.set = [_batch_fields(case, seed), torch.zeros(total, dtype=torch.float32, device=DEV)]
        initial = self.set[0].clone()
        params = (fmx.fmx_params * len(rows))()
        bufs = (fmx.fmx_buffers * len(rows))()
        for i, (nx, ny, cf, pitch, off, size) in enumerate(rows):
            params[i] = fmx.make_params((nx, ny), courant=cf, precision=fmx.FMX_F32, m=case["m"],
                                        filter_target=fmx.FMX_FILTER_NONE, pitch=pitch,
                                        stream=ctypes.c_void_p(self.stream.cuda_stream))
            for s in range(2):
                base = self.set[s].data_ptr() + 4 * off
                for c in range(3):
                    bufs[i].E[s][c] = base + 4 * c * size
                    bufs[i].B[s][c] = base + 4 * (3 + c) * size
        torch.cuda.synchronize()
        self.handle = ctypes.c_void_p()
        fmx.check(fmx.fmx_batch_create(params, len(rows), ctypes.byref(self.handle)), "fmx_batch_create")
        wb = fmx.fmx_batch_workspace_bytes(self.handle)
        self.work = torch.zeros(wb + 256, dtype=torch.uint8, device=DEV)
        fmx.check(fmx.fmx_batch_bind(self.handle, bufs, (self.work.data_ptr() + 255) // 256 * 256, wb), "fmx_batch_bind")
        fmx.check(fmx.fmx_batch_tune(self.handle, 8, None), "fmx_batch_tune")
        torch.cuda.synchronize()
        self.set[0].copy_(initial)  # the tuner advanced the grids (an even number of steps: set 0 is current)
        self.set[1].zero_()
        torch.cuda.synchronize()

    def __del__(self):
        if getattr(self, "handle", None):
            self.stream.synchronize()
            fmx.fmx_batch_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(case=case, batch=_BatchState(case, seed))
    if kind == "gradient":
        cxy, phases, theta, E0, B0, win = _gradient_inputs(case, seed)
        run_ = GaussSourceRun((case["nx"], case["ny"]), cxy, phases, case["steps"], m=case["m"], passes=case["passes"],
                              checkpoint_every=case["every"])
        leaf = lambda t: t.clone().requires_grad_(True)
        return dict(case=case, run=run_, fn=make_function(), win=win, theta=leaf(torch.from_numpy(theta)), E0=leaf(E0),
                    B0=leaf(B0))
    E, B, J = _inputs(case, seed)
    kw = dict(precision=fmx.FMX_F64 if case["f64"] else fmx.FMX_F32, courant=0.5, with_current=J is not None)
    if kind == "residual":
        kw.update(iter_mode=fmx.FMX_ITER_RESIDUAL, tol=case["tol"])
    else:
        kw.update(m=case["m"], filter_passes=case["passes"] if J is not None else 0)
    g = fmx.Grid(_shape(case), **kw)
    g.set_fields(E, B)
    if kind == "advance" and J is not None:
        g.set_current(J)
    return dict(case=case, grid=g, J=J, views={})


def _state(s):
    """The grid's own field arrays; the views of each state set are made once."""
    g = s["grid"]
    key = fmx.fmx_field_ptr(g.handle, 0)
    v = s["views"].get(key)
    if v is None:
        v = s["views"][key] = tuple(g.field_tensor(c)[..., :s["case"]["nx"]] for c in range(6))
    return v


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        fmx.check(fmx.fmx_batch_step(b.handle, case["steps"]), "fmx_batch_step")
        return b.set[0]
    if kind == "gradient":
        EN, BN = state["fn"].apply(state["theta"], state["E0"], state["B0"], state["run"], False)
        loss = 0.5 * ((EN * EN * state["win"]).sum() + (BN * BN * state["win"]).sum())
        grads = torch.autograd.grad(loss, (state["theta"], state["E0"], state["B0"]))
        return dict(E=EN.detach(), B=BN.detach(), grad_theta=grads[0], grad_E=grads[1], grad_B=grads[2])
    g = state["grid"]
    if kind == "coupled":
        g.set_current(state["J"])
    g.step(case["steps"])
    if kind != "monitor":
        return _state(state)
    g.filter(fmx.FMX_E | fmx.FMX_B, case["passes"])
    d = g.diagnostics()
    return dict(fields=_state(state), **{k: d[k] for k in ("w_scheme", "w_plain", "divb_max", "divb_l2", "gauss_max", "gauss_l2")})


# ---------------------------------------------------------------------------
# the same passes in FP64


class _Scheme:
    """The averaged-Yee step on a periodic grid of unit cells with c = 1, in FP64."""

    def __init__(self, dims, courant, f64):
        rnd = (lambda v: v) if f64 else (lambda v: float(np.float32(v)))
        self.dims, self.dt = dims, courant / math.sqrt(dims)
        k, sg = self.dt, self.dt * self.dt
        self.k, self.q, self.c6 = rnd(k), rnd(4 * math.pi * self.dt), rnd(1 / 6)
        self.a, self.aa, self.b = rnd((sg - 1) / 6), rnd((2 * sg - 1) / 36), rnd(-sg / 6)

    def d2(self, f, a):
        return torch.roll(f, -1, AX[a]) - 2 * f + torch.roll(f, 1, AX[a])

    def fwd(self, f, a):
        return torch.roll(f, -1, AX[a]) - f

    def bwd(self, f, a):
        return f - torch.roll(f, 1, AX[a])

    def alpha(self, f, a):
        return f + self.c6 * self.d2(f, a) if a < self.dims else f

    def filter(self, f, passes):
        for _ in range(passes):
            for a in range(self.dims):
                f = f + 0.25 * self.d2(f, a)
        return f

    def curl(self, F, diff, avg):
        out = []
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            r = torch.zeros_like(F[0])
            if b < self.dims:
                r = r + self.k * diff(self.alpha(F[c], c) if avg else F[c], b)
            if c < self.dims:
                r = r - self.k * diff(self.alpha(F[b], b) if avg else F[b], c)
            out.append(r)
        return out

    def apply_a(self, E):
        out = []
        for a in range(3):
            b, c = (a + 1) % 3, (a + 2) % 3
            r = torch.zeros_like(E[0])
            if b < self.dims:
                dB = self.d2(E[a], b)
                r = r + self.a * dB
                if c < self.dims:
                    r = r + self.aa * self.d2(dB, c)
            if c < self.dims:
                r = r + self.a * self.d2(E[a], c)
            for o, third in ((b, c), (c, b)):
                if a < self.dims and o < self.dims:
                    r = r + self.b * self.fwd(self.bwd(self.alpha(E[o], third), o), a)
            out.append(r)
        return out

    def step(self, E, B, J=None, passes=0, m=4, tol=None):
        dp = self.curl(B, self.bwd, True)
        if J is not None:
            dp = [d - self.q * self.filter(j, passes) for d, j in zip(dp, J)]
        x, s = dp, 0
        n2 = sum(float(d.square().sum()) for d in dp) if tol else 0.0
        while s < m if tol is None else n2 > 0.0:
            y = [d + t for d, t in zip(dp, self.apply_a(x))]
            s += 1
            r2 = sum(float((u - v).square().sum()) for u, v in zip(y, x)) if tol else 1.0
            x = y
            if tol and r2 <= tol * tol * n2:
                break
        E = [e + d for e, d in zip(E, x)]
        B = [b - r for b, r in zip(B, self.curl(E, self.fwd, False))]
        return E, B

    def diagnostics(self, E, B):
        dims = self.dims
        ce, ae = self.curl(E, self.fwd, False), self.apply_a(E)
        ws = sum(float((E[a] * (E[a] - ae[a]) + (B[a] + ce[a]) * self.alpha(B[a], a)).sum()) for a in range(3))
        wp = sum(float((E[a].square() + B[a].square()).sum()) for a in range(3))
        div = sum(self.fwd(B[a], a) for a in range(dims))
        ga = sum(self.bwd(self.alpha(self.alpha(E[a], (a + 1) % 3), (a + 2) % 3), a) for a in range(dims))
        return dict(w_scheme=ws / (8 * math.pi), w_plain=wp / (8 * math.pi), divb_max=float(div.abs().max()),
                    divb_l2=float(div.square().sum().sqrt()), gauss_max=float(ga.abs().max()),
                    gauss_l2=float(ga.square().sum().sqrt()))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        rows, total = _batch_layout(case)
        src = _batch_fields(case, seed).double()
        out = torch.zeros_like(src)
        for nx, ny, cf, pitch, off, size in rows:
            part = lambda t, c: t[off + c * size:off + c * size + pitch * ny].view(1, ny, pitch)[..., :nx]
            sc = _Scheme(2, cf, False)
            E, B = [part(src, c) for c in range(3)], [part(src, 3 + c) for c in range(3)]
            for _ in range(case["steps"]):
                E, B = sc.step(E, B, m=case["m"])
            for c in range(6):
                part(out, c).copy_((E + B)[c])
        return out
    if kind == "gradient":
        return _exact_gradient(case, seed)
    sc = _Scheme(len(_shape(case)), 0.5, case["f64"])
    E, B, J = (None if t is None else [c.double() for c in t] for t in _inputs(case, seed))
    for _ in range(case["steps"]):
        if kind == "residual":
            E, B = sc.step(E, B, tol=case["tol"])
        else:
            E, B = sc.step(E, B, J, case["passes"] if J is not None else 0, case["m"])
    if kind != "monitor":
        return tuple(E + B)
    E, B = ([sc.filter(f, case["passes"]) for f in F] for F in (E, B))
    return dict(fields=tuple(E + B), **sc.diagnostics(E, B))


def _exact_gradient(case, seed):
    cxy, phases, theta, E0, B0, win = _gradient_inputs(case, seed)
    nx, ny = case["nx"], case["ny"]
    sc = _Scheme(2, 0.5, False)
    leaf = lambda t: t.double().clone().requires_grad_(True)
    th, e0, b0 = leaf(torch.from_numpy(theta).to(DEV)), leaf(E0), leaf(B0)

    def profile(n, centre):
        d = torch.arange(n, device=DEV, dtype=torch.float64)[None, :] - torch.from_numpy(centre).to(DEV)[:, None]
        d = d - n * torch.floor(d / n + 0.5)
        return torch.exp(-d * d / 128.0)

    gx, gy = profile(nx, cxy[:, 0]), profile(ny, cxy[:, 1])
    ph = torch.from_numpy(phases).to(DEV)
    E, B = [e0[c][None] for c in range(3)], [b0[c][None] for c in range(3)]
    zero = torch.zeros_like(E[0])
    for n in range(case["steps"]):
        amp = th * torch.sin(0.2 * (n + 0.5) * sc.dt + ph)
        jz = torch.einsum("p,py,px->yx", amp, gy, gx)[None]
        E, B = sc.step(E, B, [zero, zero, jz], case["passes"], case["m"])
    EN, BN = torch.cat(E), torch.cat(B)
    w = win.double()
    loss = 0.5 * ((EN * EN * w).sum() + (BN * BN * w).sum())
    gt, ge, gb = torch.autograd.grad(loss, (th, e0, b0))
    return dict(E=EN.detach(), B=BN.detach(), grad_theta=gt.cpu(), grad_E=ge, grad_B=gb)


# ---------------------------------------------------------------------------
# what a pass cannot do without


def _flops(dims, m, passes, current):
    """Operations per cell and step: the filter as `passes` three-point passes
    per axis (an add and a multiply-add each), the source, m sweeps, the
    update and Faraday, separable stencils evaluated once per cell."""
    source, sweep, faraday = {2: (26, 36, 12), 3: (44, 112, 24)}[dims]
    return (9 * passes * dims + 6 if current else 0) + source + m * sweep + 3 + faraday


def work(case):
    kind = case["kind"]
    if kind == "batch":
        cells = sum(nx * ny for nx, ny, _ in _batch_sizes(case))
        return dict(bytes=48 * cells * case["steps"], flops=_flops(2, case["m"], 0, False) * cells * case["steps"])
    cells = case["nx"] * case["ny"] * case.get("nz", 1)
    if kind == "gradient":
        # one forward and one adjoint step: state in and out, j_z out and in on either side
        return dict(bytes=112 * cells * case["steps"],
                    flops=(2 * _flops(2, case["m"], case["passes"], True) + 4 * case["sources"]) * cells * case["steps"])
    size, dims = 8 if case["f64"] else 4, len(_shape(case))
    if kind == "residual":
        # about a dozen sweeps reach the plane waves' 1e-13, half as many 1e-5
        return dict(bytes=12 * size * cells * case["steps"],
                    flops=(_flops(2, 12 if case["f64"] else 5, 0, False) + 9 * 12) * cells * case["steps"])
    cur = kind == "coupled" or bool(case.get("current"))
    b = (15 if cur else 12) * size * cells * case["steps"]
    f = _flops(dims, case["m"], case["passes"], cur) * cells * case["steps"]
    if kind == "coupled":
        b += 3 * size * cells * case["steps"]
    if kind == "monitor":
        # the filter reads and writes the state once; the diagnostics read it
        b += 18 * size * cells
        f += (18 * case["passes"] * dims + 120) * cells
    return dict(bytes=b, flops=f)
