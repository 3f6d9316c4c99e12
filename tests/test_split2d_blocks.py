"""The FP64 Euler block recursions in float-float pairs at P = 3, 4 and with
rectangular stencils (P = 2 too): a flux depends on its block alone, not on the blocks
that happen to share a round of a CTA, and holds to FP64 accuracy over every range
that selects one of the forms.

Invariance: a periodic state moved by whole cells gives the moved result bit for bit
(dt, lambda and every stencil are the same; tiles and rounds are not, and a flux on
a tile's edge is formed by both CTAs), and so does a repeated run.

Bar: an element is formed from u and two fluxes a direction. Both evaluations of a
flux sum at most 8 x 8 weighted terms per order over 7 orders; in 1D each is within
3 x 2^-53 of the flux scale against extended precision. 64 x 2^-53 of the component's
largest |u| + 2 lambda_x |f| + 2 lambda_y |g| leaves a margin of ten."""
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


def _state(kind, nx, ny, amp, seed=3):
    rng = np.random.default_rng(seed)
    x, y = W.centres(nx, 0.0, 1.0)[None, :], W.centres(ny, 0.0, 1.0)[:, None]
    if kind == "bump":  # steep in the middle, flat outside: every form in one tile
        w = amp * np.exp(-((x - 0.45) ** 2 + (y - 0.55) ** 2) / 0.012)
        return W.prim_to_cons_2d(1.0 + w, 0.3 + 0.5 * w, -0.2 + w, 0.8 + w)
    wave = lambda: amp * np.sin(2 * np.pi * (x + rng.uniform())) * np.cos(2 * np.pi * (y + rng.uniform()))  # noqa: E731
    return W.prim_to_cons_2d(1.0 + wave(), 0.3 + wave(), -0.2 + wave(), 0.7 * (1.0 + wave()))


def _kw(P, rect, nx, ny):
    return dict(flux=W.EULER2D, P=P, nx=nx, ny=ny, bc=W.PERIODIC, cfl=0.4, x0=0.0, x1=1.0, y0=0.0, y1=1.0,
                rect_2d=rect)


@pytest.mark.parametrize("P,rect", [(2, 1), (3, 0), (3, 1), (4, 0), (4, 1)])
@pytest.mark.parametrize("kind,nx,ny,log2amp", [("bump", 64, 52, -2), ("wave", 64, 50, -5), ("wave", 40, 37, -9)])
def test_flux_depends_on_its_block_alone(env, P, rect, kind, nx, ny, log2amp):
    torch, O, acat = env
    u0 = torch.from_numpy(_state(kind, nx, ny, 2.0 ** log2amp)).cuda()

    def one(u):
        with acat.Context(**_kw(P, rect, nx, ny)) as ctx:
            out = torch.empty_like(u)
            ctx.acat_step(u.contiguous(), out)
            torch.cuda.synchronize()
            assert ctx.acat_status() == 0
        return out

    first = one(u0)
    for dy, dx in ((0, 0), (0, 1), (1, 0), (5, 3), (7, 11)):
        moved = one(torch.roll(u0, (dy, dx), (1, 2)))
        assert torch.equal(torch.roll(moved, (-dy, -dx), (1, 2)), first), (dy, dx)


@pytest.mark.parametrize("P,rect", [(2, 0), (2, 1), (3, 0), (3, 1), (4, 0), (4, 1)])
@pytest.mark.parametrize("kind,nx,ny,log2amp", [("bump", 64, 52, -2), ("wave", 40, 37, -2), ("wave", 64, 50, -5),
                                                ("wave", 33, 29, -9), ("wave", 40, 31, -12), ("wave", 33, 26, -20),
                                                ("wave", 26, 25, -40)])
def test_step_over_the_increment_ranges_2d(env, P, rect, kind, nx, ny, log2amp):
    torch, O, acat = env
    u0 = _state(kind, nx, ny, 2.0 ** log2amp)
    out = torch.empty(u0.shape, dtype=torch.float64, device="cuda")
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    orders = torch.zeros(ny * (nx + 1) + (ny + 1) * nx, dtype=torch.int8, device="cuda")
    with acat.Context(**_kw(P, rect, nx, ny)) as ctx:
        ctx.acat_step(torch.from_numpy(u0).cuda(), out, -1.0, None, dt, orders)
        torch.cuda.synchronize()
        assert ctx.acat_status() == 0
    pr = O.Problem(**_kw(P, rect, nx, ny))
    ref, _, ox, oy = O.step_2d(pr, u0, float(dt.item()))
    oref = np.r_[ox.ravel(), oy.ravel()]
    assert np.array_equal(orders.cpu().numpy(), oref) and (oref == P).any()
    rho, mx, my, E = u0
    v, w = mx / rho, my / rho
    p = 0.4 * (E - 0.5 * (mx * v + my * w))
    big = lambda q: np.abs(np.stack(q)).max(axis=(1, 2))  # noqa: E731
    f, g = big([mx, mx * v + p, mx * w, v * (E + p)]), big([my, my * v, my * w + p, w * (E + p)])
    lx, ly = float(dt.item()) / pr.dx, float(dt.item()) / pr.dy
    scale = (big(list(u0)) + 2 * lx * f + 2 * ly * g)[:, None, None]
    err = np.abs(out.cpu().numpy() - ref) / scale
    assert err.max() <= 64 * EPS, err.max() / EPS
