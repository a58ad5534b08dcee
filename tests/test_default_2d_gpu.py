"""The default kernel of FP64 planes: the whole-step exact-sum kernel where its tiles are one wave, the FP64 stencil on
the other planes of up to 80,000 sites (one thread per site on narrow ones, else the tiles), the exact-sum tiles on
larger ones.  The default's result is bit for bit that of the variant it names; F alone takes the FP64 stencil on every
plane of up to 80,000 sites."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,variant", [((3, 3), 2), ((100, 100), 2), ((256, 256), 2), ((273, 273), 2), ((274, 274), 1),
                                           ((282, 282), 1), ((200, 400), 1), ((400, 200), 1), ((100, 700), 0),
                                           ((700, 100), 0), ((12, 5000), 0), ((128, 624), 0), ((129, 620), 1), ((5, 6000), 1), ((16000, 5), 1), ((200, 401), 2), ((300, 300), 2)])
@pytest.mark.parametrize("order", [2, 4])
def test_default_kernel_of_an_fp64_plane(shape, variant, order):
    y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(np.pi * x) * np.sin(np.pi * y)) * np.exp(0.1j * np.cos(np.pi * (x + y)))
    h, a, s = 0.3, 0.7, -1.0
    V = W.random_potential(shape, 5, 0.1)
    dt = 0.2 * max_dt(2, h, a, order, 0.1, 2.0)
    out = []
    for chosen in (None, variant):
        g = Integrator(psi, h, a, s, V, "msd", order, "c128")
        if chosen is not None:
            g.set_kernel(chosen)
        assert g.kernel_in_use() == variant
        g.step(19, dt)
        g.sync()
        out.append(g.numpy())
        g.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("shape,variant", [((3, 3), 1), ((3, 4800), 1), ((4800, 4), 1), ((5, 4800), 2), ((272, 272), 2), ((273, 273), 1),
                                           ((12, 5000), 0), ((282, 282), 1), ((283, 283), 2)])
def test_default_kernel_of_a_periodic_fp64_plane(shape, variant):
    g = Integrator(np.ones(shape, complex), 0.3, 0.7, -1.0, None, "periodic", 4, "c128")
    assert g.kernel_in_use() == variant


@pytest.mark.parametrize("shape", [(3, 3), (60, 60), (256, 256), (100, 700)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("order", [2, 4])
def test_rhs_of_a_small_plane_is_the_fp64_stencils(shape, bc, order):
    y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    psi = (1.0 + 0.05 * np.sin(2 * np.pi * (x + y))) * np.exp(0.1j * np.cos(2 * np.pi * (x - y)))
    V = W.random_potential(shape, 5, 0.1)
    out = []
    for chosen in (None, 1):
        g = Integrator(psi, 0.3, 0.7, -1.0, V, bc, order, "c128")
        if chosen is not None:
            g.set_kernel(chosen)
        out.append(g.rhs().cpu().numpy())
        g.close()
    assert np.array_equal(out[0], out[1])
