"""GPU: transforms of fields with empty columns or rows, at scales far from one. A one-dimensional transform of zeros has
no exponent of its own: it must not limit the resolution of the plane it lies in (against the oracle's numpy transforms).

Tolerance: a pass's unit is at most 2^-60.7 of the sum S of its inputs' magnitudes and its rounding errors add up to noise
of at most 0.6 unit times sqrt(n). With n <= 1536 and S at most sqrt(2 n) times the inputs' norm that is below 1e-15 of the
result's rms a pass; the largest of 1e5 values is five times the rms, so two passes stay below 1e-14 of the result's largest
value, which is no smaller than its rms."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [(32, 32), (8, 64), (64, 8), (216, 36), (1024, 16), (16, 1024)]
SCALES = [1.0, 1e-31, 1e-33, 1e-36, 1e-40, 1e-50, 1e-100, 1e-300, 1e100]


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available()
    from paper_2206_09878_gb300 import lmvd
    return lmvd


def hermitian(f):
    nz = f.shape[1]
    f[:, nz // 2, :] = 0
    f[:, :, -1] = 0
    f[:, :, 0] = 0.5 * (f[:, :, 0] + np.conj(np.roll(f[:, ::-1, 0], 1, axis=1)))
    return f


def spectra(kind, rng, nz, nxh):
    """A plane at each scale, and a plane of zeros."""
    f = rng.normal(size=(len(SCALES) + 1, nz, nxh)) + 1j * rng.normal(size=(len(SCALES) + 1, nz, nxh))
    kz = np.abs(np.fft.fftfreq(nz, 1.0 / nz))[:, None]
    kx = np.arange(nxh)[None, :]
    if kind == "low modes":                    # empty columns, whole CTAs of them
        f *= (kz < 4) & (kx < 3)
    elif kind == "one column":
        f *= kx == min(5, nxh - 2)
    elif kind == "last column":
        f *= kx == nxh - 2
    else:                                      # columns apart by 2 to 70 binary places
        f *= 2.0 ** (-2.0 * np.minimum(kx, 35))
    f[:-1] *= np.array(SCALES)[:, None, None]
    f[-1] = 0
    return hermitian(f)


def check_planes(got, ref):
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-14 * np.abs(r).max()


@pytest.mark.parametrize("nx,nz", SIZES)
@pytest.mark.parametrize("kind", ["low modes", "one column", "last column", "decay"])
def test_inverse_of_sparse_spectra(L, nx, nz, kind):
    from oracle.transforms import to_phys
    spec = spectra(kind, np.random.default_rng(nx + nz), nz, nx // 2 + 1)
    ny = spec.shape[0]
    ref = to_phys(spec, nx, nz)
    d_spec = torch.from_numpy(spec).cuda()
    phys = torch.full(ref.shape, 7.0, dtype=torch.float64, device="cuda")
    ctx = L.Context(L.lmvd_default_config(nx, ny, nz))
    L.lmvd_inverse_transform(ctx.h, d_spec, phys, 1)
    ctx.synchronize()
    check_planes(phys.cpu().numpy(), ref)
    phys.fill_(7.0)
    L.lmvd_inverse_transform_noalloc(nx, ny, nz, d_spec, phys, 1)
    torch.cuda.synchronize()
    check_planes(phys.cpu().numpy(), ref)
    ctx.close()


@pytest.mark.parametrize("nx,nz", SIZES)
@pytest.mark.parametrize("kind", ["two rows", "odd pairs", "last row", "decay"])
def test_forward_of_fields_with_empty_rows(L, nx, nz, kind):
    from oracle.transforms import to_spec
    rng = np.random.default_rng(nx * nz)
    ny, px, pz = len(SCALES) + 1, 3 * nx // 2, 3 * nz // 2
    phys = rng.normal(size=(ny, pz, px))
    row = np.arange(pz)[:, None]
    if kind == "two rows":                     # one of a pair, and one pair
        phys *= (row == 1) | (row // 2 == 2)
    elif kind == "odd pairs":
        phys *= (row // 2) % 2
    elif kind == "last row":
        phys *= row == pz - 1
    else:
        phys *= 2.0 ** (-2.0 * np.minimum(row, 35))
    phys[:-1] *= np.array(SCALES)[:, None, None]
    phys[-1] = 0
    spec = torch.full((ny, nz, nx // 2 + 1), 7.0, dtype=torch.complex128, device="cuda")
    ctx = L.Context(L.lmvd_default_config(nx, ny, nz))
    L.lmvd_forward_transform(ctx.h, torch.from_numpy(phys).cuda(), spec, 1)
    ctx.synchronize()
    check_planes(spec.cpu().numpy(), to_spec(phys, nx, nz))
    ctx.close()
