"""GPU: the transforms' block fixed-point arithmetic (64-bit integers with one exponent per 1D transform) at the
edges of its plans and of its range, against the oracle's numpy transforms.

Tolerance: a pass's unit is at most 2^-60.4 sum(|re| + |im|) <= 2^-60.4 sqrt(2) n max|x|, and its rounding errors add
up as noise of about half a unit times sqrt(n): at n = 1536 below 2^-50 of the result's rms per pass, so 1e-13 of the
largest result leaves a factor of ten even for the largest of 1e6 values."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available()
    from paper_2206_09878_gb300 import lmvd
    return lmvd


def spectra(kind, rng, ny, nz, nxh):
    f = rng.normal(size=(ny, nz, nxh)) + 1j * rng.normal(size=(ny, nz, nxh))
    if kind == "one mode":
        f *= 1e-13
        f[:, min(1, nz - 1), min(1, nxh - 2)] = 1.0
    elif kind == "wide":      # magnitudes over 60 decades inside every column
        f *= 10.0 ** (-60 * rng.random(size=f.shape))
    elif kind == "zero columns":
        f[:, :, ::2] = 0.0
    elif kind == "zero planes":
        f[1:] = 0.0
    elif kind == "planes apart":  # neighbouring planes 200 decades apart (both ranges in one launch)
        f *= 10.0 ** (200.0 * (np.arange(ny) % 3 - 1))[:, None, None]
    elif kind != "white":
        f *= float(kind)
    f[:, nz // 2, :] = 0
    f[:, :, -1] = 0
    f[:, :, 0] = 0.5 * (f[:, :, 0] + np.conj(np.roll(f[:, ::-1, 0], 1, axis=1)))
    return f


def check_planes(got, ref):
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-13 * np.abs(r).max()


# transform lengths 6, 12 (a single stage), 18, 54 (6 points a thread), 24, 36, 48, 108 (no first radix-4 stage or no
# power of two), 96, 768, and the largest, 1536 (2 columns per z-pass CTA)
@pytest.mark.parametrize("nx,nz", [(4, 8), (8, 4), (12, 36), (16, 24), (72, 32), (64, 512), (1024, 16), (16, 1024)])
@pytest.mark.parametrize("kind", ["white", "one mode", "wide", "zero columns", "zero planes", "planes apart", "1e-300",
                                  "1e-38", "1e-31", "1e18", "1e300"])
def test_both_directions(L, nx, nz, kind):
    from oracle.transforms import to_phys, to_spec
    ny = 10
    rng = np.random.default_rng(nx * 1000 + nz)
    ctx = L.Context(L.lmvd_default_config(nx, ny, nz))
    spec = spectra(kind, rng, ny, nz, nx // 2 + 1)
    phys = torch.zeros((ny, 3 * nz // 2, 3 * nx // 2), dtype=torch.float64, device="cuda")
    L.lmvd_inverse_transform(ctx.h, torch.from_numpy(spec).cuda(), phys, 1)
    back = torch.zeros((ny, nz, nx // 2 + 1), dtype=torch.complex128, device="cuda")
    L.lmvd_forward_transform(ctx.h, phys, back, 1)
    ctx.synchronize()
    ref = to_phys(spec, nx, nz)
    check_planes(phys.cpu().numpy(), ref)
    check_planes(back.cpu().numpy(), to_spec(phys.cpu().numpy(), nx, nz))
    ctx.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_inputs_stay_in_their_plane(L, bad):
    nx, ny, nz = 24, 10, 16
    ctx = L.Context(L.lmvd_default_config(nx, ny, nz))
    spec = spectra("white", np.random.default_rng(1), ny, nz, nx // 2 + 1)
    spec[3, 2, 1] = bad
    spec[5, nz // 2, 1] = bad       # Nyquist slots are ignored
    spec[6, 1, nx // 2] = bad
    phys = torch.zeros((ny, 3 * nz // 2, 3 * nx // 2), dtype=torch.float64, device="cuda")
    L.lmvd_inverse_transform(ctx.h, torch.from_numpy(spec).cuda(), phys, 1)
    back = torch.zeros((ny, nz, nx // 2 + 1), dtype=torch.complex128, device="cuda")
    L.lmvd_forward_transform(ctx.h, phys, back, 1)
    ctx.synchronize()
    fin = torch.isfinite(phys).flatten(1)
    assert fin.any(1).tolist() == fin.all(1).tolist() == [i != 3 for i in range(ny)]
    kept = torch.isfinite(torch.view_as_real(back))[:, :, :nx // 2].flatten(2)
    assert not kept[3, 0].any() and kept[[i for i in range(ny) if i != 3]].all()
    ctx.close()


# chunks of the intermediate: ten fields on grids where those take at most 512 MiB (16 x 10 x 16 and, just below, 256
# x 62 x 256 with 465), four beyond (256 x 70 x 256: 525); field counts around both
@pytest.mark.parametrize("nx,ny,nz,counts", [(16, 10, 16, (1, 4, 9, 10, 11, 21)), (256, 62, 256, (10, 11)),
                                             (256, 70, 256, (4, 5, 9))])
def test_chunks_of_fields(L, nx, ny, nz, counts):
    """Fields of one call against the same fields one call each (another plan may be picked by their number, so the
    results agree to the passes' rounding, not bit for bit)."""
    gen = torch.Generator(device="cuda").manual_seed(nx + ny)
    ctx = L.Context(L.lmvd_default_config(nx, ny, nz))
    px, pz, nxh = 3 * nx // 2, 3 * nz // 2, nx // 2 + 1
    for n in counts:
        phys = torch.randn((n, ny, pz, px), generator=gen, dtype=torch.float64, device="cuda")
        spec = torch.zeros((n, ny, nz, nxh), dtype=torch.complex128, device="cuda")
        out = torch.zeros_like(phys)
        one_s, one_p = torch.zeros_like(spec[0]), torch.zeros_like(phys[0])
        torch.cuda.synchronize()
        L.lmvd_forward_transform(ctx.h, phys, spec, n)
        L.lmvd_inverse_transform(ctx.h, spec, out, n)
        for f in range(n):
            L.lmvd_forward_transform(ctx.h, phys[f], one_s, 1)
            L.lmvd_inverse_transform(ctx.h, spec[f], one_p, 1)
            ctx.synchronize()
            assert (spec[f] - one_s).abs().max() <= 1e-13 * one_s.abs().max(), (n, f)
            assert (out[f] - one_p).abs().max() <= 1e-13 * one_p.abs().max(), (n, f)
    ctx.close()
