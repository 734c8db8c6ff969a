"""The cap on Newton's iterations holds for the reduced model in the FP32 form.

A solve that does not converge within newton_maxit steps fails and is counted, in
the FP32 form (whose early steps otherwise run in FP32, under caps of their own)
as in FP64 plain. Caps on both sides of the one from which the FP32 steps are
used give the same flow.
"""
import numpy as np
import pytest

from paper_2009_13426_gb300 import flows

pytestmark = pytest.mark.gpu

NX, NY = 40, 24


@pytest.fixture(scope="module")
def alb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2009_13426_gb300 import alb as m
    return m


def fields():
    return flows.shear_layer(NX, ny=NY, mach=1.2, T_cold=0.5, T_ratio=1.5, delta=3.0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("cap", [1, 2])
def test_small_cap_fails(alb, precision, cap):
    fl = alb.Flow(NX, NY, nu=1e-3, moments=4, precision=precision, newton_maxit=cap)
    with pytest.raises(alb.AlbError) as ei:
        fl.init(*fields())
    assert ei.value.code == alb.ALB_ENEWTON
    assert fl.stats()["newton_failures"] > 0
    fl.close()


def test_caps_around_the_mixed_solve_agree(alb):
    out = []
    for cap in (36, 37, 50):
        fl = alb.Flow(NX, NY, nu=1e-3, moments=4, precision=alb.ALB_FP32_FORM, newton_maxit=cap)
        fl.init(*fields())
        fl.step(3)
        fl.sync()
        st = fl.stats()
        assert (st["fp32_iterations"] > 0) == (cap >= 37)
        assert (st["newton_iterations"] > 0) == (cap < 37)
        out.append(np.stack(fl.moments()))
        fl.close()
    assert np.array_equal(out[1], out[2])
    assert np.abs(out[0] - out[1]).max() <= 1e-5 * np.abs(out[0]).max()
