"""3D FP32 columns kernel and the one-thread-per-site kernel: the tiled variant must give the per-site kernel's bits
on grids with one deep site, partial tiles, odd rows (no TMA), several chunks of planes, and the smallest walls."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(5, 5, 5), (5, 6, 39), (9, 12, 37), (40, 13, 70), (70, 21, 33), (6, 45, 5)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0"])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64"])
def test_columns_equal_per_site_bitwise(shape, bc, order, dtype):
    z, y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(np.pi * x) * np.sin(np.pi * y) * np.sin(np.pi * z)) * np.exp(0.1j * np.cos(np.pi * (x + y - z)))
    h, a, s = 0.3, 0.7, -1.0
    for V in (None, W.random_potential(shape, 5, 0.1)):
        dt = 0.2 * max_dt(3, h, a, order, 0.1, 2.0)
        out = []
        for variant in (0, 1):
            g = Integrator(psi, h, a, s, V, bc, order, dtype)
            g.set_kernel(variant)
            g.step(3, dt)
            g.step(16, dt)
            g.sync()
            out.append(g.numpy())
            g.close()
        assert np.array_equal(out[0], out[1]), V is None
