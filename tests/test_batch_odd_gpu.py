"""Odd step counts of a batch end in a copy back into every run's Psi: one large run, many tiny ones, both together, and
narrow runs (tiles of 32 columns) must match the runs integrated alone, bit for bit."""
import numpy as np
import pytest

from paper_1203_1263_gb300.integrator import BatchIntegrator, Integrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(1501, 903)], [(3, 3)] * 40 + [(5, 17)] * 300, [(1200, 800), (3, 4), (64, 64)],
                                    [(2000, 9)] * 12 + [(900, 33), (60, 34)]])
@pytest.mark.parametrize("steps", [1, 3])
def test_odd_counts_reach_every_site(shapes, steps):
    dt = 0.2 * max_dt(2, 0.3, 0.7, 4, 0.0, 2.0)
    runs = []
    for i, n in enumerate(shapes):
        y, x = np.meshgrid(*[np.arange(k) / k for k in n], indexing="ij")
        psi = (1.0 + 0.05 * np.sin(np.pi * x) * np.sin(np.pi * y)) * np.exp(0.1j * np.cos(np.pi * (x - y)) + 0.01j * i)
        runs.append(dict(psi0=psi, h=0.3, a=0.7, s=-1.0, dt=dt, bc="msd", order=4))
    b = BatchIntegrator(runs)
    b.step(steps)
    b.sync()
    for i in range(0, len(runs), max(1, len(runs) // 7)):
        g = Integrator(runs[i]["psi0"], 0.3, 0.7, -1.0, None, "msd", 4, "c64")
        g.step(steps, dt)
        assert np.array_equal(b.numpy(i), g.numpy()), i
        g.close()
    b.close()
