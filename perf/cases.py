"""Workloads of libfwi that performance is judged on: what a reconstruction
program has the library do, from single operator applications on the smallest
grids to whole batches of the largest ones.

A case names a call (``kind``), a grid, an array and a frequency set:

  apply     one application of K, A = I - K diag(m) or A^H to a batch of vectors
  forward   fields and data of every transmit and frequency at a tissue model
  adjoint   adjoint fields of every transmit and frequency for given sources
  gradient  misfit and gradient at the homogeneous starting model (the first
            iteration of every reconstruction)
  jacobian  J a and J^H y at the fields of the homogeneous background
  admm      one ADMM-TV iteration (Gauss-Newton m-step by CG, shrink, dual)
  step      gradient and ADMM-TV iteration, one after the other

The grids, arrays and frequency sets are those of ``phantoms.py`` (64^2 disc,
256^2 thyroid, 384^2 plane-wave acquisition, 512^2 aperture, 160 x 160 x 128
volume, the serving stream's 64-192 elements on 128^2 ... 96^3) and sizes
between them.
"""
import math

import numpy as np
import torch

from paper_2604_15796_gb300 import libfwi, phantoms

C0 = 1540.0
CG_ITERS = 10
# weights of the order the benchmark scales them to (rho about 1e-2 |J^H J|)
ADMM = dict(lam=1e-3, rho=0.1, gamma=1e-3, n_cg=CG_ITERS)
# 0.5 dB/cm/MHz, the usual attenuation of soft tissue, in Np/m/Hz
TISSUE_ALPHA = 0.5 / 8.685889638 * 100.0 * 1e-6


def _case(kind, shape, elements, freqs, pitch_mm=0.2, h_mm=None, f_lo=0.3, f_hi=None, **kw):
    """The serving stream's rules for what is not given: pixels that keep the
    aperture inside the grid, at least 3.85 of them per wavelength."""
    shape = tuple(shape)
    if h_mm is None:
        h_mm = max(0.05, elements * pitch_mm / shape[-1])
    if f_hi is None:
        f_hi = min(5.0, C0 / (3.85 * h_mm * 1e-3) * 1e-6)
    c = dict(kind=kind, nz=shape[0], ny=shape[1] if len(shape) == 3 else 0, nx=shape[-1],
             elements=elements, freqs=freqs, pitch_mm=pitch_mm, h_mm=round(h_mm, 6), f_lo=f_lo,
             f_hi=round(f_hi, 6), fp64=False, lossy=False, plane_waves=0, inv_factor=1, op="")
    c.update(kw)
    return c


def listed():
    def named(name, *a, **kw):
        return dict(_case(*a, **kw), name=name)
    return [
        # one operator application on the smallest configuration (a user's own
        # Krylov method, a check of the adjoint identity): launches and latency
        named("apply_64", "apply", (64, 64), 32, 1, 0.3, 0.15, 1.0, 1.0, op="A"),
        # the smallest forward simulation: 64^2 disc, 32 elements, 1 MHz
        named("forward_64", "forward", (64, 64), 32, 1, 0.3, 0.15, 1.0, 1.0),
        # the FP64 reference configuration: gradient and ADMM-TV step on the disc's grid
        named("fp64_step_64", "step", (64, 64), 32, 1, 0.3, 0.15, 1.0, 1.0, fp64=True),
        # forward simulation of an ordinary small serving request
        named("forward_128", "forward", (128, 128), 100, 4),
        # thyroid-like workload: 256^2, 128 elements x 6 frequencies 0.5-3 MHz
        named("forward_256", "forward", (256, 256), 128, 6, 0.2, 0.1, 0.5, 3.0),
        # adjoint solves on a grid deeper than wide, an odd number of elements
        named("adjoint_320x192", "adjoint", (320, 192), 97, 3, f_lo=0.5),
        # the 2-D plane-wave acquisition: 384^2, 64 elements x 15 frequencies,
        # 60 plane waves; first gradient of a reconstruction
        named("gradient_384_pw", "gradient", (384, 384), 64, 15, 0.78, 0.13, 0.2, 3.0,
              plane_waves=60),
        # the large aperture: 512^2, 192 elements x 12 frequencies 0.3-5 MHz
        named("forward_512", "forward", (512, 512), 192, 12, 0.2, 0.08, 0.3, 5.0),
        # a serving request's volume, attenuating background
        named("forward_96_3d", "forward", (96, 96, 96), 64, 2, lossy=True),
        # the volume: 160 x 160 x 128, 64 transmits batched, two frequencies
        named("forward_volume", "forward", (128, 160, 160), 64, 2, 0.2, 0.2, 0.5, 2.0),
        # implicit Jacobian products with more elements than one matrix tile,
        # as a user's own Gauss-Newton solver takes them
        named("jacobian_384", "jacobian", (384, 384), 192, 3, 0.2, 0.13, 0.5, 3.0),
        # the other half of a reconstruction's iteration: ADMM-TV step, thyroid-like
        named("admm_256", "admm", (256, 256), 128, 6, 0.2, 0.1, 0.5, 3.0),
    ]


# field samples (pixels x transmits x frequencies) of a drawn case
DRAW_MAX = 2.0e8


def draw(rng):
    kind = rng.choice(["apply", "forward", "forward", "adjoint", "gradient", "jacobian", "admm"])
    sides = [64, 96, 128, 160, 192, 256, 320, 384]
    while True:
        if rng.random() < 0.2:
            shape = tuple(rng.choice([32, 64, 96]) for _ in range(3))
        else:
            side = rng.choice(sides)
            shape = (side, side if rng.random() < 0.5 else rng.choice(sides))
        elements = int(round(math.exp(rng.uniform(math.log(16), math.log(192)))))
        freqs = int(round(math.exp(rng.uniform(0.0, math.log(12)))))
        samples = math.prod(shape) * elements * freqs
        flops = samples * elements
        if samples <= DRAW_MAX and (kind not in ("jacobian", "admm") or flops <= 1.0e10):
            break
    kw = {}
    if kind == "apply":
        kw["op"] = rng.choice(["K", "A", "AH"])
        freqs = 1
    elif kind == "gradient" and rng.random() < 0.5:
        kw["plane_waves"] = rng.randint(15, 75)
    elif kind in ("jacobian", "admm") and rng.random() < 0.3:
        kw["inv_factor"] = 2
    return _case(kind, shape, elements, freqs, 0.2, **kw)


# ---- geometry ---------------------------------------------------------------

def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case["ny"] else (case["nz"], case["nx"])


def _inv_shape(case):
    return tuple(s // case["inv_factor"] for s in _shape(case))


def _setup(case):
    shape, h = _shape(case), case["h_mm"] * 1e-3
    elem = phantoms.array_positions(case["elements"], case["pitch_mm"] * 1e-3, h, len(shape))
    freqs = (np.linspace(case["f_lo"], case["f_hi"], case["freqs"]) * 1e6 if case["freqs"] > 1
             else np.array([case["f_hi"] * 1e6]))
    angles = (np.deg2rad(np.linspace(-60.0, 60.0, case["plane_waves"]))
              if case["plane_waves"] else None)
    return shape, h, elem, freqs, angles


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(gen, size, dtype):
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(tuple(size) + (2,), generator=gen, device="cuda",
                                             dtype=real))


def _tissue(case, seed):
    """Speed of sound of a phantom: texture and two cysts."""
    shape, h, elem, freqs, _ = _setup(case)
    width = min(s * h for s in shape) * 1e3
    w = phantoms.tissue_phantom(shape, h, case["elements"], case["pitch_mm"] * 1e-3, freqs, seed,
                                sigma=8.0 if len(shape) == 3 else 10.0,
                                inclusions=[1520.0, 1580.0],
                                semi_mm=(0.06 * width, 0.15 * width))
    return torch.from_numpy(np.ascontiguousarray(w.sos)).cuda()


def _contrast(case, seed):
    """m = kappa / kappa0 - 1 of the phantom (kappa ~ 1/c^2, or with the
    background's attenuation everywhere)."""
    sos = _tissue(case, seed)
    if not case["lossy"]:
        return (C0 * C0 / (sos * sos) - 1.0).to(torch.complex128)
    bg = complex(1.0 / C0 ** 2, TISSUE_ALPHA / (math.pi * C0))
    return torch.complex(1.0 / (sos * sos), TISSUE_ALPHA / (math.pi * sos)) / bg - 1.0


def _model(case, seed):
    """A model part way through a reconstruction, on the inversion mesh."""
    r = case["inv_factor"]
    return _contrast(case, seed)[tuple(slice(None, None, r) for _ in _shape(case))].contiguous()


def _wavenumbers(case):
    _, _, _, freqs, _ = _setup(case)
    a0 = TISSUE_ALPHA if case["lossy"] else 0.0
    return [complex(2 * math.pi * f * np.sqrt(1.0 / C0 ** 2 + 1j * a0 / (math.pi * C0)))
            for f in freqs]


def _axes(case):
    """Pixel centres along x, [y], z."""
    shape, h, _, _, _ = _setup(case)
    t = [torch.arange(s, dtype=torch.float64, device="cuda") for s in shape]
    lateral = [(a + 0.5 - 0.5 * s) * h for a, s in zip(t[1:], shape[1:])]
    return lateral[::-1] + [t[0] * h]


def _waves(case, gen):
    """Wave fields [freq][element][grid]: a few plane waves each, of the
    frequency's wavenumber and random directions and amplitudes, as residuals
    propagated back into the medium are."""
    axes, dtype = _axes(case), torch.complex128 if case["fp64"] else torch.complex64
    out = torch.empty((case["freqs"], case["elements"]) + _shape(case), dtype=dtype, device="cuda")
    for l, k in enumerate(_wavenumbers(case)):
        d = torch.randn((8, len(axes)), generator=gen, device="cuda", dtype=torch.float64)
        d = d / d.norm(dim=1, keepdim=True)
        e = [torch.exp(1j * k.real * d[:, i:i + 1] * a).to(dtype) for i, a in enumerate(axes)]
        amp = _normal(gen, (case["elements"], 8), dtype)
        if len(axes) == 2:
            out[l] = torch.einsum("eq,qz,qx->ezx", amp, e[1], e[0])
        else:
            out[l] = torch.einsum("eq,qz,qy,qx->ezyx", amp, e[2], e[1], e[0])
    return out


def _data(case, gen, dtype):
    rows = case["plane_waves"] or case["elements"]
    return 1e-3 * _normal(gen, (case["freqs"], rows, case["elements"]), dtype)


# ---- the calls --------------------------------------------------------------

def _tv_inputs(case, seed):
    """Model, TV variables and gradient as they stand after some iterations."""
    gen = _gen(seed)
    m = _model(case, seed)
    g = _grad_op(m)
    u = 0.1 * g.abs().mean() * _normal(gen, g.shape, torch.complex128)
    grad = 3e-4 * _normal(gen, m.shape, torch.complex128)
    return m, g, u, grad


def prepare(case, seed):
    shape, h, elem, freqs, angles = _setup(case)
    dtype = torch.complex128 if case["fp64"] else torch.complex64
    gen = _gen(seed)
    n_rhs = case["elements"] * case["freqs"]
    ctx = libfwi.Context(shape, h, C0, elem, freqs,
                         precision=libfwi.FWI_FP64 if case["fp64"] else libfwi.FWI_MIXED,
                         tol=1e-10 if case["fp64"] else 1e-6, tx_angles=angles,
                         inv_factor=case["inv_factor"],
                         alpha0=TISSUE_ALPHA if case["lossy"] else 0.0)
    s = dict(kind=case["kind"], ctx=ctx)
    if case["kind"] == "apply":
        s.update(op=case["op"], m=_contrast(case, seed), v=_normal(gen, (n_rhs,) + shape, dtype))
    elif case["kind"] == "forward":
        s.update(m=_contrast(case, seed), fields=ctx.empty_fields(), data=ctx.empty_data())
    elif case["kind"] == "adjoint":
        s.update(m=_contrast(case, seed), src=_waves(case, gen), lam=ctx.empty_fields())
    elif case["kind"] == "gradient":
        m = torch.zeros(shape, dtype=torch.complex128, device="cuda")
        s.update(m=m, d_obs=_data(case, gen, dtype), grad=torch.empty_like(m))
    elif case["kind"] == "jacobian":
        ctx.forward(torch.zeros(_inv_shape(case), dtype=torch.complex128, device="cuda"))
        s.update(a=_model(case, seed), y=_data(case, gen, torch.complex128))
    elif case["kind"] == "admm":
        ctx.forward(torch.zeros(_inv_shape(case), dtype=torch.complex128, device="cuda"))
        m, g, u, grad = _tv_inputs(case, seed)
        s.update(m=m, g=g, u=u, grad=grad)
    elif case["kind"] == "step":
        m = _contrast(case, seed)
        g, u = ctx.admm_init(m)
        s.update(m=m, g=g, u=u, grad=torch.empty_like(m), d_obs=_data(case, gen, dtype),
                 data=ctx.empty_data())
    return s


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "apply":
        return ctx.apply(s["op"], s["v"], 0, None if s["op"] == "K" else s["m"])
    if kind == "forward":
        ctx.forward(s["m"], fields=s["fields"], data=s["data"])
        return {"fields": s["fields"], "data": s["data"]}
    if kind == "adjoint":
        ctx.adjoint(s["m"], s["src"], s["lam"])
        return s["lam"]
    if kind == "gradient":
        misfit, _, _ = ctx.gradient(s["m"], s["d_obs"], s["grad"])
        return {"grad": s["grad"], "misfit": misfit}
    if kind == "jacobian":
        return {"Ja": ctx.jac_forward(s["a"]), "JHy": ctx.jac_adjoint(s["y"])}
    # the last iterate is kept beside the new one, as for a checkpoint
    m, g, u = s["m"].clone(), s["g"].clone(), s["u"].clone()
    sos = torch.empty(m.shape, dtype=torch.float64, device="cuda")
    out = {"m": m, "g": g, "u": u, "sos": sos}
    if kind == "step":
        misfit, _, _ = ctx.gradient(m, s["d_obs"], s["grad"], data=s["data"])
        out.update(grad=s["grad"], data=s["data"], misfit=misfit)
    ctx.admm_tv_step(m, g, u, s["grad"], sos=sos, **ADMM)
    return out


def work(case):
    """Inputs read once, outputs written once; nominal flops (5 n log2 n per
    transform on the doubled lattice, 8 per complex multiply-add).  A solve is
    counted as three BiCGSTAB iterations, two operator applications each."""
    shape = _shape(case)
    n, n_inv = math.prod(shape), math.prod(_inv_shape(case))
    ne, nf, nt = case["elements"], case["freqs"], case["plane_waves"] or case["elements"]
    e = 16 if case["fp64"] else 8
    field, data = ne * nf * n, nf * nt * ne
    lat = math.prod(2 * s for s in shape)
    apply1 = 2 * 5.0 * lat * math.log2(lat)
    contract = 8.0 * field * ne
    kind = case["kind"]
    if kind == "apply":
        return {"bytes": 2 * field * e + 16 * n + lat * e, "flops": field / n * apply1}
    if kind == "forward":
        return {"bytes": 2 * field * e + data * e + 16 * n + nf * lat * e,
                "flops": field / n * 6 * apply1 + contract}
    if kind == "adjoint":
        return {"bytes": 2 * field * e + 16 * n + nf * lat * e, "flops": field / n * 6 * apply1}
    cg = CG_ITERS * 2 * contract
    if kind == "gradient":
        # at the homogeneous model one application per solve shows it solved
        return {"bytes": field * e + data * e + 32 * n + nf * lat * e,
                "flops": field / n * 2 * apply1 + 2 * contract}
    if kind == "jacobian":
        return {"bytes": field * e + 32 * n_inv + 32 * data, "flops": 2 * contract}
    tv = (2 * 2 * len(shape) + 3) * 16 * n_inv
    if kind == "admm":
        return {"bytes": field * e + tv, "flops": cg}
    return {"bytes": field * e + 2 * data * e + tv + nf * lat * e,
            "flops": field / n * 12 * apply1 + 2 * contract + cg}


# ---- the same results in 64 bits, by plain torch ----------------------------

def _grad_op(m):
    """Forward differences along x, [y], z, zero on the last slice."""
    out = torch.zeros((m.dim(),) + tuple(m.shape), dtype=m.dtype, device=m.device)
    for q in range(m.dim()):
        ax = m.dim() - 1 - q
        out[q].narrow(ax, 0, m.shape[ax] - 1).copy_(torch.diff(m, dim=ax))
    return out


def _grad_op_t(a):
    out = torch.zeros_like(a[0])
    for q in range(a.shape[0]):
        ax = a.shape[0] - 1 - q
        n = out.shape[ax]
        low = a[q].narrow(ax, 0, n - 1)
        out.narrow(ax, 1, n - 1).add_(low)
        out.narrow(ax, 0, n - 1).sub_(low)
    return out


def _hankel0(x):
    """H0^(1)(x): torch's Bessel functions up to 1 (beyond that they are only
    good to 4e-7), else sqrt(2 / (pi x)) e^{i (x - pi/4)} times the mean of
    (1 + i s^2 / (2 x))^{-1/2} over a Gaussian e^{-s^2}, by the trapezoidal rule
    (steps of 0.2 leave 1e-14 from x = 1 on)."""
    re, im = torch.full_like(x, 0.5), torch.zeros_like(x)
    for j in range(1, 33):
        y = (0.2 * j) ** 2 / (2.0 * x)
        r = torch.sqrt(1.0 + y * y)
        c = torch.sqrt(0.5 * (r + 1.0))
        w = math.exp(-(0.2 * j) ** 2)
        re += w * c / r
        im -= w * y / (2.0 * r * c)
    amp = 0.4 / math.pi * torch.sqrt(2.0 / x)
    far = torch.complex(re, im) * torch.polar(amp, x - 0.25 * math.pi)
    z = x.clamp(max=1.0)
    near = torch.complex(torch.special.bessel_j0(z), torch.special.bessel_y0(z))
    return torch.where(x <= 1.0, near, far)


def _green(k, r, dim):
    if dim == 2:
        return 0.25j * _hankel0(k.real * r)
    return torch.exp(1j * k * r) / (4.0 * math.pi * r)


class _Exact:
    """One frequency of a case: spectrum of the cell-integrated Green's
    function on the doubled lattice, incident fields, solves."""

    def __init__(self, case, k):
        shape, h, elem, _, _ = _setup(case)
        self.shape, self.k, self.dim = shape, k, len(shape)
        off = []
        for n in shape:
            i = torch.arange(2 * n, dtype=torch.float64, device="cuda")
            off.append(torch.where(i < n, i, i - 2 * n) * h)
        r = torch.sqrt(sum(g * g for g in torch.meshgrid(*off, indexing="ij")))
        zero = r == 0
        r[zero] = 1.0
        if self.dim == 2:
            a = h / math.sqrt(math.pi)
            ka = torch.tensor(k.real * a, dtype=torch.float64)
            j1, y1 = float(torch.special.bessel_j1(ka)), float(torch.special.bessel_y1(ka))
            f = 1j * math.pi * a / (2.0 * k)
            lat = f * j1 * (-4j) * _green(k, r, 2)
            lat[zero] = f * complex(j1, y1) - 1.0 / (k * k)
        else:
            a = h * (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0)
            ka = k * a
            vol = 4.0 * math.pi * complex(np.sin(ka) - ka * np.cos(ka)) / k ** 3
            lat = vol * _green(k, r, 3)
            lat[zero] = ((1.0 - 1j * ka) * complex(np.exp(1j * ka)) - 1.0) / (k * k)
        for ax, n in enumerate(shape):
            lat.select(ax, n).zero_()
        self.spec = torch.fft.fftn(lat) * (k * k)
        self.spec32 = self.spec.to(torch.complex64)
        self.k2dv = k * k * h ** self.dim
        self.per = max(1, int(2.0e8 // lat.numel()))  # right-hand sides at a time
        self.axes, self.elem = _axes(case), elem

    def incident(self, e0, e1):
        d = [a[None, :] - torch.as_tensor(self.elem[e0:e1, i], device="cuda")[:, None]
             for i, a in enumerate(self.axes)]
        if self.dim == 2:
            r2 = d[1][:, :, None] ** 2 + d[0][:, None, :] ** 2
        else:
            r2 = (d[2][:, :, None, None] ** 2 + d[1][:, None, :, None] ** 2
                  + d[0][:, None, None, :] ** 2)
        return _green(self.k, torch.sqrt(r2), self.dim)

    def incident_all(self):
        n = len(self.elem)
        return torch.cat([self.incident(i, min(n, i + 16)) for i in range(0, n, 16)])

    def K(self, w):
        ax = tuple(range(1, 1 + self.dim))
        spec = self.spec if w.dtype == torch.complex128 else self.spec32
        f = torch.fft.fftn(w, s=[2 * n for n in self.shape], dim=ax)
        f = torch.fft.ifftn(f.mul_(spec), dim=ax)
        return f[(slice(None),) + tuple(slice(0, n) for n in self.shape)].contiguous()

    def A(self, v, m):
        return v - self.K(m.to(v.dtype) * v)

    def solve(self, b, m, tol=1e-12):
        """A x = b for b [B][grid]: corrections by BiCGSTAB in single
        precision, residuals in 64 bits."""
        ax = tuple(range(1, b.dim()))

        def dot(u, v):
            return (u.conj() * v).to(torch.complex128).sum(dim=ax, keepdim=True)

        norm = torch.linalg.vector_norm(b, dim=ax, keepdim=True)
        x, r = torch.zeros_like(b), b.clone()
        for _ in range(8):
            size = torch.linalg.vector_norm(r, dim=ax, keepdim=True)
            if float((size / norm).max()) <= tol:
                break
            q = (r / size).to(torch.complex64)
            rh, p, d = q.clone(), q.clone(), torch.zeros_like(q)
            rho = dot(rh, q)
            for _ in range(40):
                v = self.A(p, m)
                al = rho / dot(rh, v)
                s = q - al.to(q.dtype) * v
                t = self.A(s, m)
                om = dot(t, s) / dot(t, t)
                d += al.to(q.dtype) * p + om.to(q.dtype) * s
                q = s - om.to(q.dtype) * t
                if float(torch.linalg.vector_norm(q, dim=ax).max()) < 3e-6:
                    break
                new = dot(rh, q)
                p = q + ((new / rho) * (al / om)).to(q.dtype) * (p - om.to(q.dtype) * v)
                rho = new
            x += size * d
            r = b - self.A(x, m)
        return x

    def solve_all(self, m, rhs):
        """rhs(i, j): right-hand sides i .. j - 1, for every element."""
        n = len(self.elem)
        return torch.cat([self.solve(rhs(i, min(n, i + self.per)), m)
                          for i in range(0, n, self.per)])


def _flat(f):
    return f.reshape(f.shape[0], -1)


def _weights(case):
    """Plane-wave weights [freq][transmit][element], or None."""
    _, _, elem, _, angles = _setup(case)
    if angles is None:
        return None
    x = torch.as_tensor(elem[:, 0], device="cuda")
    sn = torch.as_tensor(np.sin(angles), device="cuda")
    return [torch.exp(1j * k.real * sn[:, None] * x[None, :]) for k in _wavenumbers(case)]


def _prolong(case, a):
    for ax in range(a.dim()):
        a = a.repeat_interleave(case["inv_factor"], dim=ax)
    return a


def _restrict(case, z):
    r, s = case["inv_factor"], z.shape
    z = z.reshape([v for n in s for v in (n // r, r)])
    return z.sum(dim=tuple(range(1, 2 * len(s), 2)))


class _Jacobian:
    def __init__(self, case, fields, k2dv):
        self.case, self.f, self.k2dv, self.w = case, fields, k2dv, _weights(case)

    def J(self, a):
        af = _prolong(self.case, a).reshape(1, -1)
        y = torch.stack([c * (_flat(f) * af) @ _flat(f).T for f, c in zip(self.f, self.k2dv)])
        return y if self.w is None else torch.stack([w @ v for w, v in zip(self.w, y)])

    def JH(self, y):
        z = 0
        for l, (f, c) in enumerate(zip(self.f, self.k2dv)):
            b = y[l] if self.w is None else self.w[l].conj().T @ y[l]
            fc = _flat(f).conj()
            z = z + c.conjugate() * (fc * (b @ fc)).sum(dim=0)
        return _restrict(self.case, z.reshape(_shape(self.case)))


def _admm_exact(J, m, g, u, grad, lam, rho, gamma, n_cg):
    def normal(a):
        return J.JH(J.J(a)) + rho * _grad_op_t(_grad_op(a)) + gamma * a

    b = -grad + rho * _grad_op_t(g + u - _grad_op(m)) - gamma * m
    x, r, d = torch.zeros_like(b), b.clone(), b.clone()
    rr = (r.abs() ** 2).sum()
    for _ in range(n_cg):
        q = normal(d)
        al = rr / (d.conj() * q).sum().real
        x, r = x + al * d, r - al * q
        new = (r.abs() ** 2).sum()
        d, rr = r + (new / rr) * d, new
    m = m + x
    gm = _grad_op(m)
    a = gm - u
    size = torch.sqrt((a.abs() ** 2).sum(dim=0))
    g = a * torch.where(size > 0, torch.clamp(1.0 - (lam / rho) / size, min=0.0), 0.0)
    return m, g, u + rho * (g - gm), C0 / torch.sqrt(1.0 + m.real)


def exact(case, seed):
    kind, gen = case["kind"], _gen(seed)
    ex = [_Exact(case, k) for k in _wavenumbers(case)]
    k2dv = [e.k2dv for e in ex]
    dtype = torch.complex128 if case["fp64"] else torch.complex64
    if kind == "apply":
        v = _normal(gen, (case["elements"] * case["freqs"],) + _shape(case), dtype)
        m = _contrast(case, seed)
        out = []
        for i in range(0, v.shape[0], ex[0].per):
            w = v[i:i + ex[0].per].to(torch.complex128)
            if case["op"] == "K":
                out.append(ex[0].K(w))
            elif case["op"] == "A":
                out.append(ex[0].A(w, m))
            else:  # (I - K diag(m))^H v = v - conj(m K conj(v))
                out.append(w - (m * ex[0].K(w.conj().resolve_conj())).conj())
        return torch.cat(out)
    if kind == "forward":
        m = _contrast(case, seed)
        fields = torch.empty((case["freqs"], case["elements"]) + _shape(case),
                             dtype=torch.complex128, device="cuda")
        data = []
        for l, e in enumerate(ex):
            fields[l] = e.solve_all(m, e.incident)
            data.append(e.k2dv * (_flat(fields[l]) * m.reshape(1, -1))
                        @ _flat(e.incident_all()).T)
        return {"fields": fields, "data": torch.stack(data)}
    if kind == "adjoint":
        m, src = _contrast(case, seed), _waves(case, gen)
        return torch.stack([
            e.solve_all(m, lambda i, j: src[l, i:j].to(torch.complex128).conj().resolve_conj())
            .conj().resolve_conj() for l, e in enumerate(ex)])
    if kind == "gradient":
        d = _data(case, gen, dtype).to(torch.complex128)
        J = _Jacobian(case, [e.incident_all() for e in ex], k2dv)
        return {"grad": J.JH(-d), "misfit": 0.5 * float((d.abs() ** 2).sum())}
    if kind in ("jacobian", "admm"):
        J = _Jacobian(case, [e.incident_all() for e in ex], k2dv)
        if kind == "jacobian":
            return {"Ja": J.J(_model(case, seed)), "JHy": J.JH(_data(case, gen, torch.complex128))}
        m, g, u, grad = _tv_inputs(case, seed)
        m, g, u, sos = _admm_exact(J, m, g, u, grad, **ADMM)
        return {"m": m, "g": g, "u": u, "sos": sos}
    m = _contrast(case, seed)
    d = _data(case, gen, dtype).to(torch.complex128)
    f = [e.solve_all(m, e.incident) for e in ex]
    J = _Jacobian(case, f, k2dv)
    data = torch.stack([e.k2dv * (_flat(p) * m.reshape(1, -1)) @ _flat(e.incident_all()).T
                        for e, p in zip(ex, f)])
    # grad = J^H (F(m) - d): the receivers sit at the transmitters
    grad = J.JH(data - d)
    out = {"grad": grad, "data": data, "misfit": 0.5 * float(((data - d).abs() ** 2).sum())}
    m, g, u, sos = _admm_exact(J, m, _grad_op(m), torch.zeros_like(_grad_op(m)), grad, **ADMM)
    out.update(m=m, g=g, u=u, sos=sos)
    return out
