"""The 2D FP32 whole step on periodic planes whose tiles lie away from the ends of the rows, at one end, and around
both: bit for bit the one-thread-per-site kernel's result."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(130, 300), (41, 96), (300, 79), (7, 81), (520, 530), (3, 2000)])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64"])
def test_periodic_whole_step_equals_per_site_bitwise(shape, order, dtype):
    y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(2 * np.pi * (x + 2 * y) + 0.4)) * np.exp(0.1j * np.cos(2 * np.pi * (x - y)))
    h, a, s = 0.3, 0.7, -1.0
    V = W.random_potential(shape, 5, 0.1)
    dt = 0.2 * max_dt(2, h, a, order, 0.1, 2.0)
    out = []
    for variant, tile in ((0, -1), (1, -1), (1, 0), (1, 1), (1, 2), (1, 3)):
        g = Integrator(psi, h, a, s, V, "periodic", order, dtype)
        g.set_kernel(variant, tile)
        g.step(5, dt)
        g.sync()
        out.append(g.numpy())
        g.close()
    assert all(np.array_equal(o, out[0]) for o in out[1:])


@pytest.mark.parametrize("shape", [(900, 500), (3, 20000), (4, 12001), (30000, 3)])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64"])
def test_rhs_and_steps_of_large_and_long_periodic_planes(shape, order, dtype):
    y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(2 * np.pi * (x + 2 * y) + 0.4)) * np.exp(0.1j * np.cos(2 * np.pi * (x - y)))
    dt = 0.2 * max_dt(2, 0.3, 0.7, order, 0.0, 2.0)
    out = []
    for variant in (0, 1):
        g = Integrator(psi, 0.3, 0.7, -1.0, None, "periodic", order, dtype)
        g.set_kernel(variant)
        F = g.rhs().cpu().numpy()
        g.step(19, dt)
        g.sync()
        out.append((F, g.numpy()))
        g.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
