"""Square block recursions of the FP32 2D step at P = 3, 4 on small grids, every
value compared: profiles linear in x and y, whose indicators accept the highest order
wherever the stencil does not meet the boundary.

Bar: the pair's low part keeps the update to the rounding of the float flux
increments: at most 2^-24 for each of the two directions' sums and their products,
on increments below the largest |u|, taken twice: 2^-22 of the largest |u|."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [3, 4])
@pytest.mark.parametrize("nx,ny,bc", [(9, 9, 0), (9, 9, 1), (13, 11, 1), (19, 18, 0)])
def test_square_blocks_on_linear_profiles(P, nx, ny, bc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_2007_01416_gb300 import acat, build
    build.build()
    O.build()
    x, y = W.centres(nx, 0.0, 1.0)[None, :], W.centres(ny, 0.0, 1.0)[:, None]
    u0 = W.prim_to_cons_2d(1.0 + 0.2 * x + 0.1 * y, 0.3 - 0.1 * x + 0.2 * y, 0.2 + 0.1 * x - 0.05 * y,
                           0.9 + 0.15 * x + 0.1 * y)
    kw = dict(flux=W.EULER2D, P=P, nx=nx, ny=ny, bc=bc, cfl=0.4, x0=0.0, x1=1.0, y0=0.0, y1=1.0)
    pair = acat.to_pair(np.ascontiguousarray(u0))
    u = acat.from_pair(pair)
    orders = torch.zeros(ny * (nx + 1) + (ny + 1) * nx, dtype=torch.int8, device="cuda")
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    with acat.Context(**kw, precision=acat.PREC_F32) as ctx:
        out = torch.empty(pair.shape, dtype=torch.float32, device="cuda")
        ctx.acat_step(torch.from_numpy(np.ascontiguousarray(pair)).cuda(), out, -1.0, None, dt, orders)
        torch.cuda.synchronize()
        assert ctx.acat_status() == 0
    ref, _, ox, oy = O.step_2d(O.Problem(**kw), u, float(dt.item()))
    oref = np.r_[ox.ravel(), oy.ravel()]
    assert np.array_equal(orders.cpu().numpy(), oref) and (oref == P).any()
    err = np.abs(acat.from_pair(out.cpu().numpy()) - ref)
    assert err.max() <= 2.0 ** -22 * np.abs(u).max(), err.max()
