"""The FP32 block recursion of the 2D high-order and rectangular steps against the
oracle where its task slots differ: tiles that mix every order and both flux
directions (a smooth wave cut by a jump), square and rectangular blocks, one to a
few hundred tasks, ragged tiles, linear transport.

Bar: the pair's low part keeps the update to the rounding of the float flux
increments: at most 2^-24 for each of the two directions' sums and their products,
on increments below the largest |u|, taken twice: 2^-22 of the largest |u|. A
square block of order 4 that is accepted across the jump in one direction breaks
the premise (its Taylor sums pass |u|; with the 40 x 26 state the scheme itself
leaves the physical states), so with square blocks of the Euler equations the
values are compared where no block reaches the jump, and elsewhere the orders and
the reported status."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [W.EULER2D, W.LINEAR])
@pytest.mark.parametrize("P,rect", [(2, 1), (3, 0), (3, 1), (4, 0), (4, 1)])
@pytest.mark.parametrize("nx,ny,bc", [(9, 9, 0), (17, 33, 1), (40, 26, 0), (61, 16, 1)])
def test_block_slots_f32(flux, P, rect, nx, ny, bc):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle as O
    from paper_2007_01416_gb300 import acat, build
    build.build()
    O.build()
    x, y = W.centres(nx, 0.0, 1.0)[None, :], W.centres(ny, 0.0, 1.0)[:, None]
    wave = 0.2 * np.sin(2 * np.pi * (x + 0.1)) * np.cos(2 * np.pi * (y - 0.2)) + 0.3 * ((x > 0.6) & (y > 0.3))
    if flux == W.LINEAR:
        u0, adv = (1.0 + wave)[None], (0.8, -0.5)
    else:
        u0, adv = W.prim_to_cons_2d(1.0 + wave, 0.3 - wave, 0.2 + 0.5 * wave, 0.9 + wave), (0.0, 0.0)
    kw = dict(flux=flux, P=P, nx=nx, ny=ny, bc=bc, cfl=0.4, x0=0.0, x1=1.0, y0=0.0, y1=1.0, adv=adv, rect_2d=rect)
    pair = acat.to_pair(np.ascontiguousarray(u0))
    u = acat.from_pair(pair)
    orders = torch.zeros(ny * (nx + 1) + (ny + 1) * nx, dtype=torch.int8, device="cuda")
    dt = torch.zeros(1, dtype=torch.float64, device="cuda")
    with acat.Context(**kw, precision=acat.PREC_F32) as ctx:
        out = torch.empty(pair.shape, dtype=torch.float32, device="cuda")
        ctx.acat_step(torch.from_numpy(np.ascontiguousarray(pair)).cuda(), out, -1.0, None, dt, orders)
        torch.cuda.synchronize()
        status = ctx.acat_status()
    pr = O.Problem(**kw)
    ref, _, ox, oy = O.step_2d(pr, u, float(dt.item()))
    assert np.array_equal(orders.cpu().numpy(), np.r_[ox.ravel(), oy.ravel()])
    physical = flux == W.LINEAR or bool(
        (ref[0] > 0.0).all() and (ref[3] - 0.5 * (ref[1] ** 2 + ref[2] ** 2) / ref[0] > 0.0).all())
    assert status == (0 if physical else 1)
    keep = np.ones((ny, nx), bool)
    if flux == W.EULER2D and not rect:
        inside = (x > 0.6) & (y > 0.3)
        for dy in range(-P - 1, P + 2):
            for dx in range(-P - 1, P + 2):
                jy, jx = np.arange(ny)[:, None] + dy, np.arange(nx)[None, :] + dx
                jy, jx = (jy % ny, jx % nx) if bc == W.PERIODIC else (np.clip(jy, 0, ny - 1), np.clip(jx, 0, nx - 1))
                keep &= inside[jy, jx] == inside
    err = np.abs(acat.from_pair(out.cpu().numpy()) - ref)[:, keep]
    assert keep.sum() == 0 or err.max() <= 2.0 ** -22 * np.abs(u).max(), err.max()
