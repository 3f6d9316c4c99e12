"""The FP64 flux recursion in float-float pairs against the oracle over every
range that selects one of its forms: increments of 2^-2 (FP64 evaluation), of
2^-5..2^-8 (pairs), to 2^-10 (leading terms in pairs), around 2^-12 (float
remainders), 2^-20 and 2^-40 (float from a middle order on), states at rest and in units far from 1 (beyond the
pairs' exponent range at 1e-18 and 1e18), grids whose tiles are ragged.

Bar: an element is formed from u_i, lambda F_{i-1/2} and lambda F_{i+1/2}. Both
evaluations of a flux are sums of at most 8 x 8 weighted terms per order over 7
orders; measured against extended precision each is within 3 x 2^-53 of the flux
scale. 64 x 2^-53 of |u_i| + lambda (|F_{i-1/2}| + |F_{i+1/2}|), plus the same of
the component's largest |u| for components near zero (a momentum at rest has a
flux p of order one), holds with a margin of ten."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    O.build()
    from paper_2007_01416_gb300 import acat, build
    build.build()
    return torch, O, acat


def _state(flux, nx, amp, unit, seed):
    rng = np.random.default_rng(seed)
    x = W.centres(nx, 0.0, 1.0)
    wave = lambda: np.sin(2 * np.pi * (rng.integers(1, 3) * x + rng.uniform()))  # noqa: E731
    if flux == W.BURGERS:
        return unit * (0.4 + amp * wave())[None, :]
    rho, v, p = 1.0 + amp * wave(), rng.choice([0.0, 0.3]) + amp * wave(), 0.7 * (1.0 + amp * wave())
    return W.prim_to_cons_1d(unit * rho, v, unit * p)


@pytest.mark.parametrize("flux", [W.EULER1D, W.BURGERS])
@pytest.mark.parametrize("P", [2, 3, 4])
@pytest.mark.parametrize("nx,log2amp,unit", [(33, -2, 1.0), (97, -3, 1.0), (333, -2, 1.0), (1001, -1, 1.0),
                                             (777, -6, 1e5), (1500, -12, 1.0), (700, -4, 1.0), (2500, -5, 1.0), (401, -40, 1.0), (256, -5, 1e-12),
                                             (256, -5, 1e-18), (256, -5, 1e18), (12001, -2, 1.0), (40001, -3, 1.0)])
def test_step_over_the_increment_ranges(env, flux, P, nx, log2amp, unit):
    torch, O, acat = env
    u0 = _state(flux, nx, 2.0 ** log2amp, unit, seed=nx + P)
    kw = dict(flux=flux, P=P, nx=nx, bc=W.PERIODIC, cfl=0.4, x0=0.0, x1=1.0)
    u, out = torch.from_numpy(u0).cuda(), torch.empty(u0.shape, dtype=torch.float64, device="cuda")
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    orders = torch.zeros(nx + 1, dtype=torch.int8, device="cuda")
    with acat.Context(**kw) as ctx:
        ctx.acat_step(u, out, -1.0, None, dt, orders)
        torch.cuda.synchronize()
        assert ctx.acat_status() == 0
    pr = O.Problem(**kw)
    ref, _, oref = O.step_1d(pr, u0, float(dt.item()))
    assert np.array_equal(orders.cpu().numpy(), oref)
    lam = float(dt.item()) / pr.dx
    F = np.abs(O.fluxes_1d_at(pr, u0, float(dt.item()), np.arange(nx + 1, dtype=np.int32))[0].reshape(nx + 1, -1)).T
    scale = np.abs(u0) + lam * (F[:, :-1] + F[:, 1:]) + np.abs(u0).max(axis=1, keepdims=True)
    err = np.abs(out.cpu().numpy() - ref) / scale
    assert err.max() <= 64 * EPS, (err.max() / EPS, np.unravel_index(err.argmax(), err.shape))
