"""Small FP64 planes: the whole-step exact-sum kernel is as close to the solution of the scheme in extended precision as
the FP64 stencil is.  Both errors are sums of one rounding each per site, stage and term; over the 500 sites or more and
24 steps here they differ by a few percent, unless a rounding is common to all sites and steps (in s, V or dt scaled by
a coefficient, say), which adds up coherently."""
import numpy as np
import pytest

from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu
L, C = np.longdouble, np.clongdouble


def reference(psi, V, h, a, s, order, dt, steps):
    h, a, s, dt = L(h), L(a), L(s), L(dt)

    def F(p):
        lap = 0
        for k in (0, 1):
            one = np.roll(p, 1, k) + np.roll(p, -1, k)
            lap = lap + (one - 2 * p if order == 2 else (16 * one - np.roll(p, 2, k) - np.roll(p, -2, k) - 30 * p) / L(12))
        N = s * (p.real * p.real + p.imag * p.imag) - V
        return 1j * (a / (h * h) * lap + N * p)

    p, V = psi.astype(C), V.astype(L)
    for _ in range(steps):
        k1 = F(p)
        k2 = F(p + dt / 2 * k1)
        k3 = F(p + dt / 2 * k2)
        k4 = F(p + dt * k3)
        p = p + dt / 6 * (k1 + 2 * (k2 + k3) + k4)
    return p


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("h,a,s", [(0.2, 1.0, 1.0), (25.0 / 57.0, 0.5, -1.0), (0.31, 0.7, -0.9), (25.0 / 69.0, 0.5, -1.1)])
@pytest.mark.parametrize("shape", [(26, 31), (58, 43)])
def test_error_is_that_of_the_fp64_stencil(shape, h, a, s, order):
    y, x = np.meshgrid(*[2 * np.pi * np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.3 + 0.3 * np.sin(x) * np.cos(y)) * np.exp(1j * np.sin(x + 2 * y))
    V = 1.7 + 1.1 * np.cos(x) + 0.7 * np.sin(y)
    dt = 0.8 * max_dt(2, h, a, order, 3.5, 2.6)
    ref = reference(psi, V, h, a, s, order, dt, 24)
    err = []
    for variant in (1, 2):
        g = Integrator(psi, h, a, s, V, "periodic", order, "c128")
        g.set_kernel(variant)
        g.step(24, dt)
        g.sync()
        err.append(float(np.linalg.norm((g.numpy().astype(C) - ref).ravel().view(L)) /
                         np.linalg.norm(ref.ravel().view(L))))
        g.close()
    assert err[0] < 2e-15 and err[1] <= 1.15 * err[0], err
