"""GPU: rounding errors of the fixed-point transforms against transforms in extended precision (numpy long double), for
white inputs at several amplitudes (the unit follows the amplitude in steps of two) and in both directions."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

AMPLITUDES = (1.0, 1.15, 1.32, 1.52, 1.74)


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available()
    assert np.finfo(np.longdouble).eps < 2e-19
    from paper_2206_09878_gb300 import lmvd
    return lmvd


def reference_inverse(spec, nx, nz):
    px, pz, h, n2 = 3 * nx // 2, 3 * nz // 2, nx // 2, nz // 2
    pad = np.zeros((pz, px // 2 + 1), np.clongdouble)
    pad[:n2, :h] = spec[:n2, :h]
    pad[pz - n2 + 1:, :h] = spec[n2 + 1:, :h]
    return np.fft.irfft(np.fft.ifft(pad, axis=0, norm="forward"), n=px, axis=1, norm="forward")


def reference_forward(phys, nx, nz):
    pz, h, n2 = 3 * nz // 2, nx // 2, nz // 2
    full = np.fft.fft(np.fft.rfft(phys.astype(np.longdouble), axis=1, norm="forward"), axis=0, norm="forward")
    out = np.zeros((nz, h + 1), np.clongdouble)
    out[:n2, :h] = full[:n2, :h]
    out[n2 + 1:, :h] = full[pz - n2 + 1:, :h]
    return out


def errors(L, nx, nz, forward, seed=5):
    """Per plane (one amplitude each): the error at every point over the result's rms."""
    rng = np.random.default_rng(seed)
    ny, na = 12, len(AMPLITUDES)
    px, pz, nxh = 3 * nx // 2, 3 * nz // 2, nx // 2 + 1
    ctx = L.Context(L.lmvd_default_config(nx, ny, nz))
    amp = np.array(AMPLITUDES)[:, None, None]
    if forward:
        src, dst = np.zeros((ny, pz, px)), np.zeros((ny, nz, nxh), np.complex128)
        src[:na] = amp * rng.normal(size=(na, pz, px))
    else:
        src, dst = np.zeros((ny, nz, nxh), np.complex128), np.zeros((ny, pz, px))
        f = amp * (rng.normal(size=(na, nz, nxh)) + 1j * rng.normal(size=(na, nz, nxh)))
        f[:, nz // 2, :] = 0
        f[:, :, -1] = 0
        f[:, :, 0] = 0.5 * (f[:, :, 0] + np.conj(np.roll(f[:, ::-1, 0], 1, axis=1)))
        src[:na] = f
    d_src, d_dst = torch.from_numpy(src).cuda(), torch.from_numpy(dst).cuda()
    (L.lmvd_forward_transform if forward else L.lmvd_inverse_transform)(ctx.h, d_src, d_dst, 1)
    ctx.synchronize()
    got = d_dst.cpu().numpy()
    ctx.close()
    out = []
    for a in range(na):
        ref = (reference_forward if forward else reference_inverse)(src[a], nx, nz)
        out.append(np.abs(got[a] - ref) / np.sqrt(np.mean(np.abs(ref) ** 2)))
    return np.array(out, dtype=np.float64)


# lengths with several radix-3 stages (324, 648, 864, 972 points) beside short ones
@pytest.mark.parametrize("forward", [False, True])
@pytest.mark.parametrize("nx,nz", [(216, 36), (432, 32), (576, 24), (648, 16), (16, 648), (36, 432)])
def test_errors_do_not_pile_up(L, nx, nz, forward):
    """Rounding errors are noise: with no direction of their own the largest of 1e5 to 1e6 is about five times their rms
    (eight leaves a probability below 1e-9); a rounding with a mean adds up in a few outputs instead."""
    for e in errors(L, nx, nz, forward):
        assert e.max() <= 8 * np.sqrt(np.mean(e ** 2))


# up to 768 points; above, where the first stages carry guard bits; both mixed; a small plan (6 points a thread)
@pytest.mark.parametrize("forward", [False, True])
@pytest.mark.parametrize("nx,nz", [(32, 32), (128, 96), (512, 512), (512, 16), (16, 512), (576, 576), (768, 768), (1024, 1024),
                                   (1024, 16), (16, 1024), (648, 16), (16, 864), (864, 576)])
def test_errors_are_below_those_of_binary64(L, nx, nz, forward):
    """A binary64 radix-4/2/3 transform of white fields of these sizes has an rms error of 2.1e-16 to 3.5e-16 of the
    result's rms (3.0e-16 at 1024 x 1024). A pass's unit is at most 2^-60.7 S with S = 1.6 n rms, and its noise at most 12.4
    units at 768 points and 8 units with guard bits (a model of one transform): at most 2.1e-16 a pass at 768 points, 1.5e-16
    above, 3.0e-16 for two."""
    for e in errors(L, nx, nz, forward):
        assert np.sqrt(np.mean(e ** 2)) <= 3.0e-16
        assert e.max() <= 8 * 3.0e-16
