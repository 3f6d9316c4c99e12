"""The FP64 Euler adjoint against the oracle's complex-step Jacobian where cells
away from FL-CAT2 interfaces take the FP64 sweep (increments beyond 2^-8 of the
scales), the pairs and both in one tile, and on a grid of one tile.

Bar: an entry of J^T w sums at most 8 interfaces, each a reverse sweep of at most
7 orders of 8 x 7 products; both sides are within 4 x 2^-53 of the component's
largest entry against extended precision, and the complex step rounds alike. 64 x
2^-53 of the component's largest sum |J|^T |w| leaves a margin of eight. Cells of FL-CAT2
interfaces, whose limiter derivative is conditioned by the state, are left out;
every case keeps others."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [2, 3, 4])
@pytest.mark.parametrize("nx,log2amp,bc", [(160, -2, 0), (200, -2, 1), (120, -3, 1), (90, -4, 0), (15, -30, 0)])
def test_adjoint_away_from_limiters(P, nx, log2amp, bc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_2007_01416_gb300 import acat, build
    build.build()
    O.build()
    rng = np.random.default_rng(nx + P)
    x = W.centres(nx, 0.0, 1.0)
    wave = lambda: 2.0 ** log2amp * np.sin(2 * np.pi * (x + rng.uniform()))  # noqa: E731
    u0 = W.prim_to_cons_1d(1.0 + wave(), 0.3 + wave(), 0.7 * (1.0 + wave()))
    kw = dict(flux=W.EULER1D, P=P, nx=nx, bc=bc, cfl=0.4, x0=0.0, x1=1.0)
    pr = O.Problem(**kw)
    dt = O.dt_cfl(pr, u0)
    _, _, orders = O.step_1d(pr, u0, dt)
    w = rng.normal(size=u0.shape)
    J = np.zeros((u0.size, u0.size))
    for k in range(u0.size):
        e = np.zeros(u0.size)
        e[k] = 1e-30
        J[:, k] = O.step_1d_complex(pr, u0, e.reshape(u0.shape), dt)[1].ravel() / 1e-30
    ref = (J.T @ w.ravel()).reshape(u0.shape)
    scale = (np.abs(J).T @ np.abs(w).ravel()).reshape(u0.shape).max(axis=1, keepdims=True)
    with acat.Context(**kw) as ctx:
        out = torch.empty(u0.shape, dtype=torch.float64, device="cuda")
        ctx.acat_adjoint_step(torch.from_numpy(u0).cuda(), dt, torch.from_numpy(w).cuda(), out)
        torch.cuda.synchronize()
    keep = np.ones(nx, bool)
    for m in np.nonzero(orders == 1)[0]:
        j = np.arange(m - 2, m + 2)
        keep[j % nx if bc == W.PERIODIC else np.clip(j, 0, nx - 1)] = False
    assert keep.mean() > 0.7 and (orders == P).mean() > 0.7
    err = (np.abs(out.cpu().numpy() - ref) / scale)[:, keep]
    assert err.max() <= 64 * 2.0 ** -53, err.max() * 2.0 ** 53
