"""Counters of D2Q49: the FP32 steps of a solve are in fp32_iterations and, as in
FP64 plain, in newton_iterations."""
import pytest

pytestmark = pytest.mark.gpu


def test_d2q49_counts_its_fp32_steps():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2009_13426_gb300 import alb, flows
    out = {}
    for start in (alb.ALB_START_AUTO, alb.ALB_START_MAXWELLIAN):
        fl = alb.Flow(24, 16, nu=1e-3, stencil=49, moments=13, newton_start=start)
        fl.init(*flows.shear_layer(24, ny=16, mach=1.0, T_cold=0.5, T_ratio=1.5, delta=2.0))
        fl.step(2)
        fl.sync()
        out[start] = fl.stats()
        fl.close()
    auto, full = out[alb.ALB_START_AUTO], out[alb.ALB_START_MAXWELLIAN]
    assert full["fp32_iterations"] == 0
    assert 0 < auto["fp32_iterations"] < auto["newton_iterations"]
    assert auto["newton_calls"] == full["newton_calls"]
