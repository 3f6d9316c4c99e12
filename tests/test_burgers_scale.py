"""FP64 Burgers steps whose local |u| is far below the scale that dt suggests: a
region at 1/4 to 1/16 of the grid's largest |u|, an imposed dt of CFL / 4 to
CFL / 16, and the same dt as a step clipped at t_end. The flux recursion picks its
precision by increments against a velocity scale, which has to be the stencil's own.

Bar, in 2^-53 of V, the largest |u| of the cell's stencils: u - lambda dF is
rounded to 1 on each side, and the difference of the fluxes to less than 1/2; a flux is
within 3 of its scale V^2 / 2 on each side, two fluxes to a cell, with
lambda V <= CFL V / (div max |u|) = 0.4 scale / div. 3 + 3 scale / div."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [2, 3, 4])
@pytest.mark.parametrize("nx,scale,k,div", [(800, 1 / 16, 16, 1), (1600, 1 / 8, 4, 1), (800, 1 / 4, 16, 4),
                                            (200, 1.0, 4, 16), (1600, 1 / 16, 4, 8)])
def test_local_scale(P, nx, scale, k, div):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_2007_01416_gb300 import acat, build
    build.build()
    O.build()
    x = W.centres(nx, 0.0, 1.0)
    u0 = (np.where(x < 0.9, scale, 1.0) * (0.2 + 0.75 * np.sin(2 * np.pi * k * x + 0.2)))[None, :]
    kw = dict(flux=W.BURGERS, P=P, nx=nx, bc=W.PERIODIC, cfl=0.4, x0=0.0, x1=1.0)
    pr = O.Problem(**kw)
    dt = O.dt_cfl(pr, u0) / div
    ref, _, orders = O.step_1d(pr, u0, dt)
    assert (orders == P).mean() > 0.8
    with acat.Context(**kw) as ctx:
        u, out = torch.from_numpy(u0).cuda(), torch.empty(u0.shape, dtype=torch.float64, device="cuda")
        ctx.acat_step(u, out, dt)
        clipped = u.clone()
        ctx.acat_run(clipped, 1, dt)
        torch.cuda.synchronize()
        assert ctx.acat_status() == 0
    if div > 1:
        assert torch.equal(clipped, out)
    got = out.cpu().numpy()
    V = np.max([np.abs(np.roll(u0, s, axis=1)) for s in range(-P - 1, P + 2)], axis=0)
    err = np.abs(got - ref)[0] / V[0] * 2.0 ** 53
    err = err[(np.abs(x - 0.9) > (P + 2) / nx) & (x > (P + 2) / nx) & (x < 1 - (P + 2) / nx)]
    assert err.max() <= 3 + 3 * scale / div, err.max()


@pytest.mark.parametrize("P", [2, 3, 4])
@pytest.mark.parametrize("nx,log2amp,div", [(333, -2, 4), (777, -3, 16), (1500, -8, 64)])
def test_euler_below_cfl(P, nx, log2amp, div):
    """Euler at dt below CFL: its scales are the node's own. Bar as for the CFL dt in
    test_split_recursion.py: both fluxes within 3 x 2^-53 of the flux scale and a
    margin of ten, 64 x 2^-53 of |u_i| + lambda (|F_l| + |F_r|) and the largest |u|."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_2007_01416_gb300 import acat, build
    build.build()
    O.build()
    x = W.centres(nx, 0.0, 1.0)
    w = 2.0 ** log2amp * np.sin(2 * np.pi * x + 0.3)
    u0 = W.prim_to_cons_1d(1.0 + w, 0.3 - w, 0.7 * (1.0 + 0.5 * w))
    kw = dict(flux=W.EULER1D, P=P, nx=nx, bc=W.PERIODIC, cfl=0.4, x0=0.0, x1=1.0)
    pr = O.Problem(**kw)
    dt = O.dt_cfl(pr, u0) / div
    ref, _, orders = O.step_1d(pr, u0, dt)
    out = torch.empty(u0.shape, dtype=torch.float64, device="cuda")
    codes = torch.zeros(nx + 1, dtype=torch.int8, device="cuda")
    with acat.Context(**kw) as ctx:
        ctx.acat_step(torch.from_numpy(u0).cuda(), out, dt, None, None, codes)
        torch.cuda.synchronize()
        assert ctx.acat_status() == 0
    assert np.array_equal(codes.cpu().numpy(), orders) and (orders == P).any()
    F = np.abs(O.fluxes_1d_at(pr, u0, dt, np.arange(nx + 1, dtype=np.int32))[0].reshape(nx + 1, -1)).T
    scale = np.abs(u0) + dt / pr.dx * (F[:, :-1] + F[:, 1:]) + np.abs(u0).max(axis=1, keepdims=True)
    err = np.abs(out.cpu().numpy() - ref) / scale
    assert err.max() <= 64 * 2.0 ** -53, err.max() * 2.0 ** 53
