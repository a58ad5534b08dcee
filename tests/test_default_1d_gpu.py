"""The default route of FP64 lines around the lengths where it changes: bit for bit one thread per site."""
import numpy as np
import pytest

from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2500, 2501, 12500, 12501, 14500, 14501, 22500, 22501, 32768, 32769])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("order", [2, 4])
def test_default_line_equals_per_site_bitwise(n, bc, order):
    x = np.arange(n) / n
    psi = (1.0 + 0.1 * np.sin(40 * np.pi * x)) * np.exp(0.3j * np.cos(60 * np.pi * x))
    out = []
    for variant in (None, 3 if n > 32768 else 0):
        g = Integrator(psi, 0.3, 0.7, -1.0, None, bc, order, "c128")
        if variant is not None:
            g.set_kernel(variant)
        g.step(19, 0.2 * max_dt(1, 0.3, 0.7, order, 0.0, 2.0))
        g.sync()
        out.append(g.numpy())
        g.close()
    assert np.array_equal(out[0], out[1])
