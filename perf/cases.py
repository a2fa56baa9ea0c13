"""The calls whose time counts: RK2 steps and substages of the solver, its start-up, its gradient and its
transforms, through the public entry points, from the smallest grids to the largest.

A case is a dict of plain values; "call" says which entry point it exercises:
  step       ctx.step(1) (two substages), then ctx.get_state: a time-stepping program that reads its state
  substage   ctx.advance_substage(), then ctx.get_state (large grids, where one substage is long enough)
  startup    ctx.set_state without history (20 fixed-point applications), then dz/dt and m^c
  gradient   autograd.Substages forward and backward: the adjoint path
  inverse    lmvd_inverse_transform, `fields` fields (FP64 synthesis with the 3/2 rule)
  forward    lmvd_forward_transform
  noalloc    lmvd_inverse_transform_noalloc (no context, no device allocation)
A step moves its context on, as a program's does: the second pass on a state is the next step.
"""
import math

import torch

from paper_2206_09878_gb300 import autograd as A
from paper_2206_09878_gb300 import lmvd as L

# numbers of Fourier modes the transforms take: 3 n / 2 has no prime factors but 2 and 3
SIZES = (12, 16, 24, 32, 36, 48, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 384, 432, 512)
TRANSFORMS = ("inverse", "forward", "noalloc")
NOALLOC_BYTES = 31 << 20  # T plus twiddles of lmvd_inverse_transform_noalloc have to fit in 32 MiB


def _case(call, nx, ny, nz, precision=0, order=6, bc=0, fields=0, substages=0, side=False):
    return dict(call=call, nx=nx, ny=ny, nz=nz, precision=precision, order=order, bc=bc, fields=fields,
                substages=substages, side=side)


def listed():
    named = {
        # a quick look or a unit test of a user's program: launches, latency and short y-solves count
        "step 32": _case("step", 32, 33, 32, side=True),
        # odd sizes, another spline order, potential matching: a small physics study in double-float
        "step 72x61x48 p5 df": _case("step", 72, 61, 48, precision=1, order=5, bc=1, side=True),
        # the everyday production run, in both arithmetics
        "step 128": _case("step", 128, 129, 128, side=True),
        "step 128 df": _case("step", 128, 129, 128, precision=1, side=True),
        # the paper's own 3D mesh with its potential matching: few modes, long y-systems
        "step 128x512x128": _case("step", 128, 512, 128, bc=1),
        # a run at 256^3 in the precision path
        "substage 256 df": _case("substage", 256, 257, 256, precision=1),
        # the largest: the transform lengths and mode counts of 512^3, half of its rows
        "substage 512x257x512": _case("substage", 512, 257, 512),
        # the start-up a run pays once, and again at every restart without history
        "startup 96x81x96": _case("startup", 96, 81, 96),
        # the differentiation path: two substages forward, their adjoints backward
        "gradient 64": _case("gradient", 64, 65, 64, substages=2, side=True),
        # analysis of a user's own fields, synthesis for its output files, at ragged sizes
        "forward 256x129x256": _case("forward", 256, 129, 256, fields=3),
        "inverse 216x65x108": _case("inverse", 216, 65, 108, fields=4),
        # synthesis inside another framework that owns the device memory: one small call
        "noalloc 64x33x64": _case("noalloc", 64, 33, 64, fields=1),
    }
    return [dict(c, name=n) for n, c in named.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(("step", "step", "step", "substage", "substage", "startup", "gradient", "inverse", "forward",
                       "noalloc"))
    most = dict(step=192, substage=512, startup=144, gradient=72, inverse=512, forward=512, noalloc=128)[call]
    least = 64 if call == "substage" else 12
    while True:
        fit = [s for s in SIZES if least <= s <= most]
        nx, nz = rng.choice(fit), rng.choice(fit)
        ny = _log_int(rng, 20, dict(step=520, substage=520, startup=200, gradient=97, inverse=300, forward=300,
                                    noalloc=200)[call])
        points = nx * ny * nz
        if call == "step" and not 1e4 <= points <= 1.7e7:
            continue
        if call == "substage" and not 1e6 <= points <= 6.7e7:
            continue
        if call in ("startup", "gradient") and points > (1.2e6 if call == "startup" else 4.5e5):
            continue
        fields = rng.randint(1, 6) if call in TRANSFORMS else 0
        if fields and points * fields > 1e8:
            continue
        if call == "noalloc" and 16 * ny * (3 * nz // 2) * (nx // 2) + 48 * (nx + nz) + 1024 > NOALLOC_BYTES:
            continue
        if call in TRANSFORMS:
            return _case(call, nx, ny, nz, fields=fields)
        precision = 0 if call == "gradient" else rng.randint(0, 1)
        # six is the order in use; the others the solver takes as well
        return _case(call, nx, ny, nz, precision=precision, order=rng.choice((4, 5, 6, 6, 6, 7, 8)),
                     bc=rng.randint(0, 1), substages=rng.randint(1, 3) if call == "gradient" else 0,
                     side=points < 4e6 and rng.random() < 0.7)


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _hermitian(f):
    """Makes the kx = 0 column of spectral planes [..., nz, nxh] Hermitian in kz and the Nyquist slots zero."""
    nz, nxh = f.shape[-2:]
    f[..., nz // 2, :] = 0
    f[..., :, nxh - 1] = 0
    col = f[..., :, 0]
    f[..., :, 0] = 0.5 * (col + torch.conj(torch.roll(torch.flip(col, (-1,)), 1, -1)))
    return f


def _wavenumbers(nx, nz):
    kx = torch.arange(nx // 2 + 1, device="cuda", dtype=torch.float64)[None, :]
    kz = torch.fft.fftfreq(nz, 1.0 / nz, device="cuda", dtype=torch.float64)[:, None]
    return torch.sqrt(kx * kx + kz * kz)


def _spectral_noise(g, rows, nx, nz, kmax):
    """Random phases and amplitudes on the band 0 < |k| <= kmax, one pattern for all rows."""
    z = torch.randn((nz, nx // 2 + 1, 2), generator=g, device="cuda", dtype=torch.float64)
    k = _wavenumbers(nx, nz)
    return _hermitian(torch.view_as_complex(z) * ((k > 0) & (k <= kmax)))


def _flow(case, seed):
    """A Rayleigh-Taylor state: heavy fluid over light with a rough interface, and weak divergence-free motion."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    g = _generator(seed)
    kmax = max(2, min(nx, nz) // 16)
    ratio, width = 3.0, 0.1
    eta = torch.fft.irfft2(_spectral_noise(g, 1, nx, nz, kmax), s=(nz, nx), norm="forward")
    eta = eta * (0.01 / eta.square().mean().sqrt())
    y = torch.linspace(-1.0, 1.0, ny, device="cuda", dtype=torch.float64)
    ys = torch.linspace(-1.0, 1.0, ny + 1, device="cuda", dtype=torch.float64)
    rl = 1.0 / ratio
    z = torch.empty((ny, nz, nx // 2 + 1), device="cuda", dtype=torch.complex128)
    for a in range(0, ny, 32):  # by rows: the physical fields need not be held whole
        rho = 0.5 * (1 + rl) + 0.5 * (1 - rl) * torch.tanh((y[a:a + 32, None, None] - eta[None]) / width)
        z[a:a + 32] = torch.fft.rfft2((1.0 - rl / rho) / (1.0 - rl), norm="forward")
    z[:, nz // 2, :] = 0
    z[:, :, nx // 2] = 0
    prof1, prof2 = 1 - y ** 2, (1 - ys ** 2) ** 2
    prof1[[0, -1]] = 0
    prof2[[0, 1, -2, -1]] = 0
    k = _wavenumbers(nx, nz)
    out = dict(z=z)
    for name, prof, scale in (("om", prof1, k), ("m2", prof2, torch.ones_like(k))):
        f = _spectral_noise(g, ny, nx, nz, kmax)
        f = f * (1e-3 / f.abs().square().sum().sqrt())
        out[name] = prof[:, None, None] * (f * scale)[None]
    for name in ("mm1", "mm3"):
        out[name] = prof1 * 1e-3 * torch.randn((), generator=g, device="cuda", dtype=torch.float64)
    return out


def _config(case):
    return L.lmvd_default_config(case["nx"], case["ny"], case["nz"], precision=case["precision"], bc_mode=case["bc"],
                                 spline_order=case["order"], rho_light=1.0 / 3.0, re=1000.0, dt=1e-4)


def _spectral_fields(case, seed):
    """Smooth spectra with noise in every retained mode, as products of a flow's fields have."""
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["fields"]
    f = torch.randn((n * ny, nz, nx // 2 + 1, 2), generator=_generator(seed), device="cuda", dtype=torch.float64)
    f *= (1.0 / (1.0 + _wavenumbers(nx, nz)) ** 2)[None, :, :, None]
    return _hermitian(torch.view_as_complex(f)).reshape(n, ny, nz, nx // 2 + 1).contiguous()


def _physical_fields(case, seed):
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["fields"]
    g = _generator(seed)
    shape = (n, ny, 3 * nz // 2, 3 * nx // 2)
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    return x.mul_(0.1).add_(torch.randn((n, ny, 1, 1), generator=g, device="cuda", dtype=torch.float64))


_SIDE = []


def _side_stream():
    """One stream of the program's own for all its contexts (substages replay as CUDA graphs there)."""
    if not _SIDE:
        _SIDE.append(torch.cuda.Stream())
    return _SIDE[0]


def prepare(case, seed):
    """A context on its grid with a state loaded, or a transform's input and output fields."""
    call, nx, ny, nz, n = case["call"], case["nx"], case["ny"], case["nz"], case["fields"]
    s = dict(call=call, case=case)
    if call == "noalloc":
        s["spec"] = _spectral_fields(case, seed)
        s["phys"] = torch.empty((n, ny, 3 * nz // 2, 3 * nx // 2), device="cuda", dtype=torch.float64)
        return s
    stream = _side_stream() if case["side"] else None
    ctx = s["ctx"] = L.Context(_config(case), stream=stream)
    if call in ("inverse", "forward"):
        if call == "inverse":
            s["spec"] = _spectral_fields(case, seed)
            s["phys"] = torch.empty((n, ny, 3 * nz // 2, 3 * nx // 2), device="cuda", dtype=torch.float64)
        else:
            s["phys"] = _physical_fields(case, seed)
            s["spec"] = torch.empty((n, ny, nz, nx // 2 + 1), device="cuda", dtype=torch.complex128)
        return s
    st = _flow(case, seed)
    if call == "startup":
        s["state"] = st
    elif call == "gradient":
        s["x"] = A.state_from_dict(st)
        with torch.no_grad():
            _, hist = A.Startup.apply(s["x"], ctx)
        s["hist"] = hist.clone()
        g = _generator(seed + 1)
        s["g_x"] = torch.randn(s["x"].shape, generator=g, device="cuda", dtype=torch.float64)
        s["g_hist"] = torch.randn(hist.shape, generator=g, device="cuda", dtype=torch.float64)
        s["x"].requires_grad_(True)
        s["hist"].requires_grad_(True)
    else:
        ctx.set_state(st)
        s["out"] = ctx.empty_state()
    return s


def run(s):
    call, case = s["call"], s["case"]
    if call == "noalloc":
        L.lmvd_inverse_transform_noalloc(case["nx"], case["ny"], case["nz"], s["spec"], s["phys"], case["fields"])
        return s["phys"]
    ctx = s["ctx"]
    if call == "inverse":
        L.lmvd_inverse_transform(ctx.h, s["spec"], s["phys"], case["fields"])
        return s["phys"]
    if call == "forward":
        L.lmvd_forward_transform(ctx.h, s["phys"], s["spec"], case["fields"])
        return s["spec"]
    if call == "step":
        ctx.step(1)
        return ctx.get_state(s["out"])
    if call == "substage":
        ctx.advance_substage()
        return ctx.get_state(s["out"])
    if call == "startup":
        ctx.set_state(s["state"])
        return [ctx.field(w) for w in (L.LMVD_FIELD_ZDOT, L.LMVD_FIELD_MC1, L.LMVD_FIELD_MC2, L.LMVD_FIELD_MC3)]
    x, hist = A.Substages.apply(s["x"], s["hist"], ctx, 0, case["substages"], 2)
    gx, gh = torch.autograd.grad((x, hist), (s["x"], s["hist"]), (s["g_x"], s["g_hist"]))
    return [x.detach(), hist.detach(), gx, gh]


# ---------------------------------------------------------------- what a pass cannot do without
def _transform_flops(nx, ny, nz):
    """5 n log2 n per one-dimensional complex transform: nx/2 columns and 3nz/4 row pairs in each plane."""
    px, pz = 3 * nx // 2, 3 * nz // 2
    return ny * (nx / 2 * 5 * pz * math.log2(pz) + pz / 2 * 5 * px * math.log2(px))


def work(case):
    nx, ny, nz, p = case["nx"], case["ny"], case["nz"], case["order"]
    spec, phys = 16.0 * ny * nz * (nx // 2 + 1), 8.0 * ny * (3 * nx // 2) * (3 * nz // 2)
    ft = _transform_flops(nx, ny, nz)
    if case["call"] in TRANSFORMS:
        return dict(bytes=case["fields"] * (spec + phys), flops=case["fields"] * ft)
    # one fixed-point application: 4 syntheses and 2 analyses; two collocation solves, one solve per mode, five
    # evaluations, on complex values with about p entries a row
    points = ny * nz * (nx // 2 + 1)
    apply = 6 * ft + points * 4.0 * p * (2 + 2 + 5)
    # a substage (kf = 4): 28 syntheses, 20 analyses, about 19 solves and 30 evaluations
    substage = 48 * ft + points * 4.0 * p * (19 + 30)
    if case["call"] == "startup":
        return dict(bytes=4 * spec + 3 * spec, flops=9 * ft + 20 * apply)
    if case["call"] == "gradient":
        # state and history in and out, their adjoints in and out; the adjoint does each transform again
        n = case["substages"]
        return dict(bytes=36 * spec, flops=n * 3 * substage)
    n = 2 if case["call"] == "step" else 1
    # state and history (9 fields) read, six new fields written, the state read out
    return dict(bytes=(9 + 6 + 3) * spec, flops=n * substage)


def exact(case, seed):
    """The transforms' outputs by torch.fft on the padded grid. A whole substage has no such value here: it
    would be a second solver."""
    nx, ny, nz, n = case["nx"], case["ny"], case["nz"], case["fields"]
    px, pz, h, n2 = 3 * nx // 2, 3 * nz // 2, nx // 2, nz // 2
    if case["call"] in ("inverse", "noalloc"):
        spec = _spectral_fields(case, seed)
        out = torch.empty((n, ny, pz, px), device="cuda", dtype=torch.float64)
        for f in range(n):
            pad = torch.zeros((ny, pz, px // 2 + 1), device="cuda", dtype=torch.complex128)
            pad[:, :n2, :h] = spec[f, :, :n2, :h]
            pad[:, pz - n2 + 1:, :h] = spec[f, :, n2 + 1:, :h]
            out[f] = torch.fft.irfft2(pad, s=(pz, px), norm="forward")
        return out
    if case["call"] == "forward":
        phys = _physical_fields(case, seed)
        out = torch.zeros((n, ny, nz, nx // 2 + 1), device="cuda", dtype=torch.complex128)
        for f in range(n):
            full = torch.fft.rfft2(phys[f], norm="forward")
            out[f, :, :n2, :h] = full[:, :n2, :h]
            out[f, :, n2 + 1:, :h] = full[:, pz - n2 + 1:, :h]
        return out
    return None
