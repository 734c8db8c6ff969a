"""States on both sides of the fixed-point range, and the block shapes of FP64 plain.

The FP32 form refines in 64-bit fixed point where every exponent lies within 31
octaves (and the bound on them within 44 nepers), in FP64 beyond. The exponents
come here from the state's own multipliers, so that each case is shown to lie on
its side. FP64 plain steps small grids in blocks of 256 threads and larger ones
in blocks of 128: a node's update is the same code in both and in the batch.
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


def exponents(alb, u, T):
    """1 + lambda . P(xi_i) of the equilibrium of (u, 0, T)."""
    import torch

    def dev(v):
        return torch.tensor([v], dtype=torch.float64, device="cuda")
    feq = torch.empty(21, dtype=torch.float64, device="cuda")
    lam = torch.empty(8, dtype=torch.float64, device="cuda")
    st = torch.empty(1, dtype=torch.int32, device="cuda")
    alb.alb_equilibrium(dev(1.0), dev(u), dev(0.0), dev(T), 1, 1e-12, 50, feq, lam, None, st)
    assert int(st[0]) == 0
    x, y = (np.asarray(a, np.float64) for a in alb.alb_velocities())
    r2 = x * x + y * y
    P = np.stack([np.ones(21), x, y, x * x, x * y, y * y, x * r2, y * r2])
    return 1.0 + lam.cpu().numpy() @ P


@pytest.mark.parametrize("T,u,outside", [(0.27, 0.45, True), (0.25, 0.3, True), (0.30, 0.45, True),
                                         (0.35, 0.45, False), (0.40, 0.0, False)])
def test_both_sides_of_the_fixed_point_range(alb, T, u, outside):
    octaves = exponents(alb, u, T).max() / np.log(2.0)
    assert (octaves >= 31.0) == outside
    n = 48
    rho, jx, jy, e = flows.uniform(n, n, ux=u, T=T)
    f = 1.0 + 1e-3 * np.random.default_rng(7).uniform(-1.0, 1.0, rho.shape)
    fields = (rho * f, jx * f, jy * f, e * f)
    out = []
    for prec in (alb.ALB_FP64_PLAIN, alb.ALB_FP32_FORM):
        fl = alb.Flow(n, n, nu=1e-2, precision=prec)
        fl.init(*fields)
        fl.step(5)
        fl.sync()
        out.append(fl.moments())
        if prec == alb.ALB_FP32_FORM:
            assert fl.stats()["newton_iterations"] == 0  # the FP64 Newton is not needed
        fl.close()
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-5 * np.abs(out[0][3]).max()


@pytest.mark.parametrize("nx,ny", [(33, 7), (40, 8), (31, 13), (512, 512), (521, 505)])
def test_fp64_block_shapes_give_the_same_bits(alb, nx, ny):
    kw = dict(nu=1e-4, sensor=1, precision=alb.ALB_FP64_PLAIN)
    fields = flows.shear_layer(nx, ny=ny, delta=max(1.0, ny / 16.0))
    fl = alb.Flow(nx, ny, **kw)
    fl.init(*fields)
    fl.step(3)
    b = alb.Batch([dict(nx=nx, ny=ny, **kw)])
    try:
        for v, (block, _) in enumerate(alb.alb_batch_variants(alb.ALB_FP64_PLAIN)):
            b.set_tuning(alb.ALB_FP64_PLAIN, variant=v, tile_w=(16, 32, block))
            b.flows[0].init(*fields)
            b.step(3)
            for p, q in zip(fl.primitives() + list(fl.shifts()),
                            b.flows[0].primitives() + list(b.flows[0].shifts())):
                assert np.array_equal(p, q), v
            assert fl.stats()["reconstructions"] == b.flows[0].stats()["reconstructions"]
    finally:
        b.close()
        fl.close()
