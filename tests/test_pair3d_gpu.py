"""Small 3D FP64 grids, a lane per component: the per-site kernel must give the tiled kernel's bits (both with the
FP64 stencil) on grids with one interior cell between walls, no or one deep site, uneven sides and several blocks."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(3, 3, 3), (3, 8, 11), (4, 5, 13), (9, 3, 4), (5, 5, 5), (7, 12, 9), (11, 25, 16), (32, 32, 32)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0"])
@pytest.mark.parametrize("order", [2, 4])
def test_pair_equals_tiled_bitwise(shape, bc, order):
    z, y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(np.pi * x) * np.sin(np.pi * y) * np.sin(np.pi * z)) * np.exp(0.1j * np.cos(np.pi * (x + y - z)))
    h, a, s = 0.3, 0.7, -1.0
    for V in (None, W.random_potential(shape, 5, 0.1)):
        dt = 0.2 * max_dt(3, h, a, order, 0.1, 2.0)
        out = []
        for variant in (0, 1):
            g = Integrator(psi, h, a, s, V, bc, order, "c128")
            g.set_kernel(variant)
            r = g.rhs()
            g.step(3, dt)
            g.step(16, dt)
            g.sync()
            out.append((r.cpu().numpy(), g.numpy()))
            g.close()
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1]), V is None
