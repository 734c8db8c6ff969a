"""Solves whose FP32 phase has no finite start.

A temperature below 2^-126 is positive in FP64 and zero in FP32: the Maxwellian
start of the solvers that take their early steps in FP32 is then 0 x infinity.
Such a solve must be left to the FP64 iteration and end as it does there, never
as a converged equilibrium of NaNs.
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


def outcome(alb, T, **kw):
    """Error code, populations and primitives of an initial state at rest."""
    fl = alb.Flow(16, 16, nu=1e-3, **kw)
    code = 0
    try:
        fl.init(*flows.uniform(16, 16, T=T))
    except alb.AlbError as e:
        code = e.code
    out = list(fl.populations()) + list(fl.primitives())
    fl.close()
    return code, out


@pytest.mark.parametrize("start", ["AUTO", "PREVIOUS"])
@pytest.mark.parametrize("stencil,moments", [(21, 8), (49, 13)])
@pytest.mark.parametrize("T", [1e-39, 1e-42, 1e-60, 1e-37])
def test_temperature_below_fp32_ends_as_in_fp64(alb, T, stencil, moments, start):
    if stencil == 49 and start == "PREVIOUS":
        pytest.skip("D2Q49 starts from the Maxwellian")
    kw = dict(stencil=stencil, moments=moments)
    ref_code, ref = outcome(alb, T, newton_start=alb.ALB_START_MAXWELLIAN, **kw)
    code, got = outcome(alb, T, newton_start=getattr(alb, "ALB_START_" + start), **kw)
    assert code == ref_code
    for a, b in zip(got, ref):
        assert np.all(np.isfinite(a))
        assert np.allclose(a, b, rtol=1e-12, atol=0)


@pytest.mark.parametrize("moments", [8, 4])
@pytest.mark.parametrize("T", [1e-39, 1e-37])
def test_fp32_form_gives_no_nan(alb, T, moments):
    _, got = outcome(alb, T, precision=alb.ALB_FP32_FORM, moments=moments)
    for a in got:
        assert np.all(np.isfinite(a))
