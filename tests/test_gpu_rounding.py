"""Rounding of the FP32 form's moment sums and collision, bit for bit.

The next lattice of a node is a step function of its velocity, so a velocity
that is rounded otherwise moves nodes beside a threshold into another lattice,
which changes their results by far more than FP32's rounding. The roundings are
therefore fixed: the compensated sums (each velocity's product by its component
or |xi|^2 rounded by itself, in the order of the velocity table, then added with
Neumaier's correction), and in the collision f* = f + (f^eq - f)/tau with f^eq -
f rounded from the rounded f^eq, g* = g + (g^eq - g)/tau with g^eq - g rounded
once. The inputs are the flow's own exported populations.
"""
import numpy as np
import pytest

from paper_2009_13426_gb300 import flows

pytestmark = pytest.mark.gpu

F = np.float32
NX, NY, NU = 96, 56, 1e-3


@pytest.fixture(scope="module")
def state():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2009_13426_gb300 import alb
    rng = np.random.default_rng(11)
    y, x = np.mgrid[0:NY, 0:NX]
    wave = [0.08 * np.sin(2 * np.pi * (a * x / NX + b * y / NY) + p)
            for a, b, p in ((1, 2, 0.3), (3, -1, 1.1), (-2, 2, 2.0))]
    fields = flows.conserved(1.0 + wave[0] + 1e-3 * rng.uniform(-1, 1, x.shape), 0.15 + wave[1],
                             -0.2 + wave[2], 0.6 + wave[0])
    fl = alb.Flow(NX, NY, nu=NU, precision=alb.ALB_FP32_FORM)
    fl.init(*fields)
    fl.step(3)
    before = np.stack(fl.populations()).astype(F)
    fl.step(1)
    fl.sync()
    after = np.stack(fl.populations()).astype(F).reshape(2, 21, -1)
    prim = np.stack(fl.primitives()).astype(F).reshape(4, -1)
    assert not np.any(fl.shifts()) and not np.any(fl.next_shifts())  # no pull is rebuilt
    vx, vy = alb.alb_velocities()
    fl.close()
    pulled = np.empty_like(before)
    for i in range(21):
        pulled[:, i] = np.roll(before[:, i], (vy[i], vx[i]), axis=(1, 2))
    return pulled.reshape(2, 21, -1), after, prim, np.asarray(vx), np.asarray(vy)


class Sum:
    def __init__(self, n):
        self.s, self.c = np.zeros(n, F), np.zeros(n, F)

    def add(self, v):
        t = self.s + v
        self.c = self.c + np.where(np.abs(self.s) >= np.abs(v), (self.s - t) + v, (v - t) + self.s)
        self.s = t

    def value(self):
        return (self.s + self.c).astype(np.float64)


def test_moment_sums(state):
    (f, g), _, prim, vx, vy = state
    n = f.shape[1]
    r, jx, jy, e = Sum(n), Sum(n), Sum(n), Sum(n)
    for i in range(21):
        r.add(f[i])
        if vx[i]:
            jx.add(F(vx[i]) * f[i])
        if vy[i]:
            jy.add(F(vy[i]) * f[i])
        c2 = vx[i] ** 2 + vy[i] ** 2
        if c2:
            e.add(F(c2) * f[i])
        e.add(g[i])
    rho = r.value()
    inv = 1.0 / rho
    ux, uy = jx.value() * inv, jy.value() * inv
    T = (e.value() - rho * (ux * ux + uy * uy)) * inv * 0.2
    assert np.array_equal(rho.astype(F), prim[0])
    assert np.array_equal(ux.astype(F), prim[1])
    assert np.array_equal(uy.astype(F), prim[2])
    # (the last FP64 bit of T may differ, and with it one rounding)
    assert np.all(np.abs(T.astype(F) - prim[3]) <= np.spacing(prim[3]))


def fma(a, b, c):
    # the product is exact in FP64; rounding twice shows at one value in 2^28
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def test_relaxation(state):
    (f, g), (fs, gs), prim, _, _ = state
    rho, T = prim[0], prim[3]
    om = F(1) / (F(0.5) + F(NU) / T)
    gp = F(3) * T  # 2 Cv - D at gamma = 1.4
    found = np.zeros(f.shape, bool)
    for i in range(21):
        # the equilibrium per unit density is some FP32 number near this one
        near = (((fs[i].astype(np.float64) - f[i]) / om + f[i]) / rho).astype(F)
        for k in range(-12, 13):
            fe = (near.view(np.int32) + k).view(F) * rho
            found[i] |= (fma(om, fe - f[i], f[i]) == fs[i]) & \
                        (fma(om, fma(gp, fe, -g[i]), g[i]) == gs[i])
    assert found.mean() > 0.9999
