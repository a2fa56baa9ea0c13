"""GPU: the banded solves of grids with few modes at the edges of their row blocks (every spline order, from the fewest
rows the solver takes to a few blocks), forward against the oracle and transposed against central differences.

Tolerances: the state 1e-12 as in the parity tests (the solves are those of the oracle up to rounding); the adjoint's
directional derivative against a central difference of step 1e-5 relative: truncation ~1e-10 and rounding ~1e-15 / 1e-5
of the loss, so 1e-6."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    assert torch.cuda.is_available()
    from paper_2206_09878_gb300 import lmvd
    return lmvd


@pytest.mark.parametrize("bc", ["walls", "potential"])
@pytest.mark.parametrize("p,ny", [(4, 10), (4, 37), (5, 10), (5, 23), (6, 10), (6, 22), (7, 11), (7, 29), (8, 12), (8, 41)])
def test_state_matches_oracle(L, p, ny, bc):
    from _pairs import compare_states, make_pair, to_numpy, to_torch
    over = dict(nx=8, ny=ny, nz=8, kmax=2, p=p, width=0.3, u_rms=1e-2)
    if bc == "potential":
        over["bc"] = bc
    S, ctx, st, cfg = make_pair(L, "rt32", **over)
    S.set_state(**st)
    ctx.set_state(to_torch(st))
    for _ in range(3):
        S.advance_substage()
        ctx.advance_substage()
    gpu = to_numpy(ctx.get_state())
    ctx.synchronize()
    ctx.close()
    e = compare_states(S, gpu, S.state())
    assert all(v <= 1e-12 for v in e.values()), e


@pytest.mark.parametrize("precision", [0, 1])
def test_fields_after_the_start_up(L, precision):
    """rho_t and m^c of the last start-up application can be read and conserve mass (to rounding: an m^c of
    double-float transforms is still solved for in FP64)."""
    from _pairs import make_pair, to_torch
    S, ctx, st, cfg = make_pair(L, "rt32", precision=precision)
    ctx.set_state(to_torch(st))
    rt, m1, m2, m3 = (ctx.field(f).cpu().numpy() for f in (L.LMVD_FIELD_RHO_T, L.LMVD_FIELD_MC1, L.LMVD_FIELD_MC2,
                                                           L.LMVD_FIELD_MC3))
    ctx.close()
    for m in (m1, m2, m3):
        assert np.abs(m).max() > 0
    assert np.linalg.norm(S.mass_residual(rt, (m1, m2, m3))) <= 1e-12 * np.linalg.norm(rt)


@pytest.mark.parametrize("p,ny", [(4, 10), (5, 24), (7, 30), (8, 45)])
def test_adjoint_directional_derivative(L, p, ny):
    from _pairs import make_pair, to_torch
    from paper_2206_09878_gb300 import autograd as A
    S, ctx, st, cfg = make_pair(L, "rt32", nx=8, ny=ny, nz=8, kmax=2, p=p, width=0.3, u_rms=1e-2)
    x = A.state_from_dict(to_torch(st))
    x, hist = A.Startup.apply(x, ctx)
    x, hist = x.detach(), hist.detach()
    g = torch.Generator(device="cuda").manual_seed(p)
    w = torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)
    d = x * torch.randn(x.shape, generator=g, device="cuda", dtype=torch.float64)   # respects the zero slots

    def loss(y):
        out, _ = A.Substages.apply(y, hist, ctx, 0, 1, 1)
        return (w * out).sum()

    y = x.clone().requires_grad_(True)
    (gx,) = torch.autograd.grad(loss(y), y)
    h = 1e-5
    with torch.no_grad():
        fd = float((loss(x + h * d) - loss(x - h * d)) / (2 * h))
    ad = float((gx * d).sum())
    ctx.close()
    assert abs(fd - ad) <= 1e-6 * abs(fd), (fd, ad)
