"""nlse_rhs under every kernel variant: variants of one arithmetic give the same bits (4 runs as 1 where it is not the
fused FP32 kernel), and the two FP64 stencils agree to rounding."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(40,), (20, 31), (9, 17, 24)])
@pytest.mark.parametrize("dtype", ["c128", "c64", "c64_acc64"])
def test_rhs_of_every_variant(shape, dtype):
    g = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(2 * np.pi * sum(g))) * np.exp(0.1j * np.cos(2 * np.pi * g[0]))
    V = W.random_potential(shape, 5, 0.1)
    F = []
    for variant in range(5):
        c = Integrator(psi, 0.3, 0.7, -1.0, V, "msd", 4, dtype)
        c.set_kernel(variant)
        F.append(c.rhs().cpu().numpy())
        c.close()
    assert np.array_equal(F[0], F[1]) and np.array_equal(F[1], F[4]) and np.array_equal(F[2], F[3])
    assert np.max(np.abs(F[2] - F[0])) <= 1e-11 * np.max(np.abs(F[0]))
