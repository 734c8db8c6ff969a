"""Residual evaluations of alb_equilibrium in the FP32 form.

The FP32 Newton ends at a residual of about 1e-6 and hands its Cholesky factor to
the refinement. With the factor of that point the refinement contracts by some
1e-4 per residual, so the third residual meets 1e-12 at the latest; with a factor
one step older it needs up to five.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_three_residuals_suffice():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2009_13426_gb300 import alb
    rng = np.random.default_rng(21)
    n = 50000

    def dev(a):
        return torch.tensor(a, dtype=torch.float64, device="cuda")
    rho, T = dev(rng.uniform(0.5, 2.0, n)), dev(rng.uniform(0.45, 0.8, n))
    u, v = dev(rng.uniform(-0.5, 0.5, n)), dev(rng.uniform(-0.5, 0.5, n))
    feq = torch.empty(n * 21, dtype=torch.float64, device="cuda")
    iters = torch.empty(n, dtype=torch.int32, device="cuda")
    status = torch.empty(n, dtype=torch.int32, device="cuda")
    alb.alb_equilibrium(rho, u, v, T, n, 1e-12, 50, feq, None, iters, status,
                        precision=alb.ALB_FP32_FORM)
    torch.cuda.synchronize()
    assert not status.any()
    assert int(iters.max()) <= 3
