"""The FP64 Euler adjoint with level Jacobians in float-float pairs against the
oracle's complex-step Jacobian, over the increments that select its routes:
2^-2 of the scales (FP64 sweep), 2^-4 (mixed), 2^-9 and 2^-20 (pairs), velocity
units of 1e-5 and 1e5 (pairs) and 1e7 (enthalpy beyond the pairs' bound: FP64
sweep); grids with ragged tiles and of one tile.

Bar: an entry of J^T w sums at most 8 interfaces, each a reverse sweep of at most
7 orders of 8 x 7 products; both sides were measured within 4 x 2^-53 of the
component's largest entry against extended precision, and the complex step rounds
alike. 64 x 2^-53 of the component's largest sum |J|^T |w| leaves a margin of
eight. Cells of FL-CAT2 interfaces, whose limiter derivative is conditioned by
the state, are left to the other adjoint tests."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [2, 3, 4])
@pytest.mark.parametrize("nx,log2amp,unit,bc", [(33, -2, 1.0, 0), (40, -4, 1.0, 1), (65, -9, 1.0, 0), (48, -20, 1.0, 1),
                                                (15, -12, 1.0, 0), (65, -9, 1e-5, 0), (65, -9, 1e5, 0), (65, -9, 1e7, 0)])
def test_adjoint_over_the_increment_ranges(P, nx, log2amp, unit, bc):
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
    u0 = W.prim_to_cons_1d(1.0 + wave(), unit * (0.3 + wave()), 0.7 * unit ** 2 * (1.0 + wave()))
    kw = dict(flux=W.EULER1D, P=P, nx=nx, bc=bc, cfl=0.4, x0=0.0, x1=1.0)
    pr = O.Problem(**kw)
    dt = O.dt_cfl(pr, u0)
    _, _, orders = O.step_1d(pr, u0, dt)
    s = (unit ** np.arange(3.0))[:, None]
    w = rng.normal(size=u0.shape) / s
    # columns scaled to a unit step of each component
    J = np.zeros((u0.size, u0.size))
    for k in range(u0.size):
        e = np.zeros(u0.size)
        e[k] = 1e-30 * s[k // nx, 0]
        J[:, k] = O.step_1d_complex(pr, u0, e.reshape(u0.shape), dt)[1].ravel() / 1e-30
    ref = (J.T @ w.ravel()).reshape(u0.shape)
    scale = (np.abs(J).T @ np.abs(w).ravel()).reshape(u0.shape).max(axis=1, keepdims=True)
    with acat.Context(**kw) as ctx:
        out = torch.empty(u0.shape, dtype=torch.float64, device="cuda")
        ctx.acat_adjoint_step(torch.from_numpy(u0).cuda(), dt, torch.from_numpy(w).cuda(), out)
        torch.cuda.synchronize()
        got = out.cpu().numpy() * s
    keep = np.ones(nx, bool)
    for m in np.nonzero(orders == 1)[0]:
        j = np.arange(m - 2, m + 2)
        keep[j % nx if bc == W.PERIODIC else np.clip(j, 0, nx - 1)] = False
    err = (np.abs(got - ref) / scale)[:, keep]
    assert np.isfinite(got).all()
    assert keep.sum() == 0 or err.max() <= 64 * 2.0 ** -53, err.max() * 2.0 ** 53
