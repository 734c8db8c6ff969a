"""Launch shapes and solver branches of the step kernel.

The single-flow step picks its block by the grid's size and the batch has
shapes of its own; a node's update is the same code in all of them, so their
results must be equal bit for bit. Sizes on both sides of each choice, with
remainders of the 32 x 8 and 32 x 12 tiles. States whose exponents lie outside
the fixed-point range (cold gas, |ubar| near 1/2) take the FP64 refinement: the
FP32 form is held to its 1e-5 against FP64 plain there too.
"""
import numpy as np
import pytest

from paper_2009_13426_gb300 import flows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def alb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2009_13426_gb300 import alb as m
    return m


@pytest.mark.parametrize("nx,ny", [(33, 7), (40, 8), (31, 13), (512, 512), (521, 505), (1030, 1020)])
def test_every_block_shape_gives_the_same_bits(alb, nx, ny):
    kw = dict(nu=1e-4, sensor=1, precision=alb.ALB_FP32_FORM)
    fields = flows.shear_layer(nx, ny=ny, delta=max(1.0, ny / 16.0))
    fl = alb.Flow(nx, ny, **kw)
    fl.init(*fields)
    fl.step(3)  # (thin layers flag failed rebuilds: their fallback values are compared too)
    b = alb.Batch([dict(nx=nx, ny=ny, **kw)])
    try:
        for v in (0, 2, 4):
            b.set_tuning(alb.ALB_FP32_FORM, variant=v, tile_w=(32, 32, 32))
            b.flows[0].init(*fields)
            b.step(3)
            for p, q in zip(fl.primitives() + list(fl.shifts()),
                            b.flows[0].primitives() + list(b.flows[0].shifts())):
                assert np.array_equal(p, q), v
            s, t = fl.stats(), b.flows[0].stats()
            assert s["reconstructions"] == t["reconstructions"]
    finally:
        b.close()
        fl.close()


@pytest.mark.parametrize("T,u", [(0.27, 0.45), (0.25, 0.3), (0.35, 0.45)])
def test_cold_states_beyond_the_fixed_point_range(alb, T, u):
    n = 48
    rho, jx, jy, e = flows.uniform(n, n, ux=u, T=T)
    rng = np.random.default_rng(7)
    f = 1.0 + 1e-3 * rng.uniform(-1.0, 1.0, rho.shape)
    fields = (rho * f, jx * f, jy * f, e * f)
    out = []
    for prec in (alb.ALB_FP64_PLAIN, alb.ALB_FP32_FORM):
        fl = alb.Flow(n, n, nu=1e-2, precision=prec)
        fl.init(*fields)
        fl.step(5)
        fl.sync()
        out.append(fl.moments())
        fl.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-5 * np.abs(out[0][3]).max()
