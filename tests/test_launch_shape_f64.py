"""The launch shape of a single 1D FP64 context: the reported warps per CTA are those
of the step's kernel (4 to 8; no FP64 step has 2), applying them or a value that
earlier versions reported (8, or 2 for large grids) changes nothing, and any other is
refused; a batch runs the same states at every shape, at the largest tiles too."""
import numpy as np
import pytest

from paper_2007_01416_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2007_01416_gb300 import acat, build
    build.build()
    return torch, acat


@pytest.mark.parametrize("nx,P,stored", [(400, 2, 8), (16384, 4, 2), (262144, 2, 2), (777, 1, 8)])
def test_reported_shape(env, nx, P, stored):
    torch, acat = env
    with acat.Context(**W.euler1d_riemann_entropy(nx=nx, seed=1, P=P).problem_kwargs()) as ctx:
        shape = ctx.acat_launch_shape()
        assert 4 <= shape[0] <= 8 and shape[1:] == (1, 0)
        for nw in (shape[0], stored):
            ctx.acat_set_launch_shape(nw, 1, 0)
            assert ctx.acat_launch_shape() == shape
        with pytest.raises(acat.AcatError) as ei:
            ctx.acat_set_launch_shape(3, 1, 0)
        assert ei.value.code == -5


@pytest.mark.parametrize("flux", [W.EULER1D, W.BURGERS, W.LINEAR])
@pytest.mark.parametrize("P", [1, 2, 3])
def test_batch_shapes_f64(env, flux, P):
    torch, acat = env
    sizes = [700, 33, 1201]
    rng = np.random.default_rng(P)
    if flux == W.EULER1D:
        u0 = np.concatenate([W.euler1d_riemann_entropy(nx=n, seed=n, P=P).u0 for n in sizes], axis=1)
    else:
        u0 = np.concatenate([0.4 + 0.5 * np.sin(2 * np.pi * (W.centres(n, 0.0, 1.0) + rng.uniform())) for n in sizes])[None]
    first = None
    kw = dict(flux=flux, P=P, nx=sizes[0], bc=W.TRANSMISSIVE, cfl=0.4, x0=0.0, x1=1.0, adv=(0.7, 0.0))
    with acat.Context(**kw, sizes=sizes) as ctx:
        for nw in (8, 4, 16):
            ctx.acat_set_launch_shape(nw, 1, 0)
            u = torch.from_numpy(np.ascontiguousarray(u0)).cuda()
            ctx.acat_run(u, 5)
            torch.cuda.synchronize()
            assert ctx.acat_status() == 0
            first = u if first is None else first
            assert torch.equal(u, first), nw
