"""The solvers that steps and initial states run, on random states.

alb_equilibrium and alb_equilibrium13 run the FP64 Newton (or the refinement in
FP64); a flow's solves run the fixed-point refinement (FP32 form) or take their
early steps in FP32 (FP64 plain, D2Q49) and come to the former only where those
fail. Here every node of a flow is a state of its own: with nu = 0 Grad's factors
are one and the first collision gives 2 f^eq - f^eq, so the exported populations
are the flow's own equilibria, from a Maxwellian start and, for starts from
previous multipliers, from a warm one.

Every node's populations either meet the constraints of the state (the root is
unique) or are the zeros of a failed solve; a solve fails only where the FP64
Newton does.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NX, NY = 256, 96
N = NX * NY
CV = 2.5


@pytest.fixture(scope="module")
def alb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2009_13426_gb300 import alb as m
    return m


def states(region, seed):
    """rho, u, v, T of N nodes; u and v also choose the lattice (u_max 2)."""
    rng = np.random.default_rng(seed)
    ub, t = {"inside": (0.5, (0.32, 1.2)), "cold": (0.3, (0.24, 0.32)),
             "edge": (0.5, (0.18, 0.30)), "fast": (0.5, (0.5, 1.0))}[region]
    rho = rng.uniform(0.2, 3.0, N)
    u = rng.integers(-2, 3, N) + rng.uniform(-ub, ub, N)
    v = rng.integers(-2, 3, N) + rng.uniform(-ub, ub, N)
    if region == "fast":  # beyond the range of the outermost lattice
        u = np.sign(u) * rng.uniform(2.5, 2.6, N)
    return rho, u, v, rng.uniform(*t, N)


def solve(alb, s, **kw):
    """(f per unit density (q, N), ub, vb, T, failed) of an initial state."""
    rho, u, v, T = s
    fields = [a.reshape(NY, NX) for a in
              (rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v) + rho * CV * T)]
    fl = alb.Flow(NX, NY, nu=0.0, **kw)
    try:
        fl.init(*fields)
    except alb.AlbError as e:
        assert e.code == alb.ALB_ENEWTON
    f, _ = fl.populations()
    sx, sy = fl.shifts()
    fl.close()
    f = f.reshape(f.shape[0], N) / rho
    r, jx, jy, e = [a.reshape(N) for a in fields]
    ux, uy = jx / r, jy / r
    T = (e - 0.5 * r * (ux * ux + uy * uy)) / (r * CV)
    return f, ux - sx.reshape(N), uy - sy.reshape(N), T, ~np.any(f, axis=0)


def residual(alb, f, u, v, T, moments):
    """Largest violation of the constraints at every node."""
    vel = alb.alb_stencil_velocities(49 if moments == 13 else 21)
    x, y = (np.asarray(a, np.float64) for a in vel)
    r2, one, u2 = x * x + y * y, np.ones_like(x), u * u + v * v
    if moments == 8:
        P = [one, x, y, x * x, x * y, y * y, x * r2, y * r2]
        m = [1.0 + 0 * u, u, v, u * u + T, u * v, v * v + T, u * (u2 + 4 * T), v * (u2 + 4 * T)]
    elif moments == 4:
        P, m = [one, x, y, r2], [1.0 + 0 * u, u, v, u2 + 2 * T]
    else:
        E = 0.5 * u2 + T
        P = [one, x, y, x * x, x * y, y * y, x ** 3, x * x * y, x * y * y, y ** 3, x * x * r2,
             x * y * r2, y * y * r2]
        m = [1.0 + 0 * u, u, v, u * u + T, u * v, v * v + T, u * (u * u + 3 * T),
             (u * u + T) * v, u * (v * v + T), v * (v * v + 3 * T),
             2 * ((E + 2 * T) * u * u + (E + T) * T), 2 * (E + 2 * T) * u * v,
             2 * ((E + 2 * T) * v * v + (E + T) * T)]
    return np.abs(np.stack(P) @ f - np.stack(m)).max(0)


CASES = [("fp32", 21, 8, "AUTO"), ("fp32", 21, 8, "MAXWELLIAN"), ("fp32", 21, 4, "AUTO"),
         ("fp64", 21, 8, "AUTO"), ("fp64", 21, 8, "PREVIOUS"), ("fp64", 49, 13, "AUTO")]


@pytest.mark.parametrize("region", ["inside", "cold", "edge", "fast"])
@pytest.mark.parametrize("prec,stencil,moments,start", CASES)
def test_every_state_meets_its_constraints_or_fails_as_in_fp64(alb, prec, stencil, moments, start,
                                                               region):
    s = states(region, 5)
    kw = dict(stencil=stencil, moments=moments)
    ref = solve(alb, s, newton_start=alb.ALB_START_MAXWELLIAN, **kw)
    got = solve(alb, s, precision=alb.ALB_FP32_FORM if prec == "fp32" else alb.ALB_FP64_PLAIN,
                newton_start=getattr(alb, "ALB_START_" + start), **kw)
    f, u, v, T, failed = got
    assert np.all(np.isfinite(f))
    # a residual of 1e-12 in each of the two solves, the second one's targets formed
    # from the first one's sums (monomials up to 27, 81 on D2Q49); FP32 populations
    # round to 6e-8
    limit = 1e-5 if prec == "fp32" else 1e-10
    assert np.all(residual(alb, f[:, ~failed], u[~failed], v[~failed], T[~failed], moments)
                  <= limit)
    assert not np.any(failed & ~ref[4])  # fails only where the FP64 Newton does
    if region == "inside":
        # the same root: FP64's bound is that of the sweeps against the oracle
        both = ~failed & ~ref[4]
        assert both.mean() > 0.9
        assert np.abs(f[:, both] - ref[0][:, both]).max() <= (1e-5 if prec == "fp32" else 1e-9)
