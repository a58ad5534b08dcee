"""The 1D several-steps kernel against the one-thread-per-site kernel, which evaluates the same per-site
arithmetic from global memory: bit for bit.  Lengths: the smallest lines (one interior site), one CTA, edges and
remainders of the CTAs' own sites (the last CTA with one site or none but the wall's), many CTAs; step counts below, at and beyond one launch and one graph."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


def run(psi, V, bc, order, dtype, variant, steps):
    h, a, s = 0.3, 0.7, -1.0
    dt = 0.2 * max_dt(1, h, a, order, 0.0 if V is None else float(np.max(np.abs(V))), 2.0)
    g = Integrator(psi, h, a, s, V, bc, order, dtype)
    if variant is not None:
        g.set_kernel(variant)
    for n in steps:
        g.step(n, dt)
    g.sync()
    out = g.numpy()
    g.close()
    return out


@pytest.mark.parametrize("n", [3, 4, 5, 17, 31, 65, 129, 1000, 2001, 5003])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dtype", ["c128", "c64", "c64_acc64"])
def test_several_steps_equal_per_site_bitwise(n, bc, order, dtype):
    x = np.arange(n) / n
    psi = (1.0 + 0.05 * np.sin(np.pi * x)) * np.exp(0.1j * np.cos(np.pi * x))
    for V in (None, W.random_potential((n,), 5, 0.1)):
        for steps in ((1,), (3, 21), (37,)):
            ref = run(psi, V, bc, order, dtype, 0, steps)
            for variant in (None, 1):   # the default route and the chosen one
                assert np.array_equal(run(psi, V, bc, order, dtype, variant, steps), ref), (variant, steps, V is None)


@pytest.mark.parametrize("n,dtype", [(32768, "c128"), (120001, "c64"), (120001, "c64_acc64")])
def test_long_lines_equal_per_site_bitwise(n, dtype):
    x = np.arange(n) / n
    psi = (1.0 + 0.1 * np.sin(40 * np.pi * x)) * np.exp(0.3j * np.cos(60 * np.pi * x))
    assert np.array_equal(run(psi, None, "msd", 4, dtype, None, (20,)), run(psi, None, "msd", 4, dtype, 0, (20,)))
