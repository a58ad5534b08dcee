"""The 2D whole-step kernel (four RK4 stages of a tile in one launch) against the
one-thread-per-site kernel, which evaluates the same per-site arithmetic from
global memory: the two must agree bit for bit.  Shapes: the smallest grids (one
interior site, both walls in one tile), single tiles, tile edges and remainders
of every tile shape, grids with tiles away from every wall; step counts with
pairs, an odd step through the copy, and graph replays with a remainder."""
import numpy as np
import pytest

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu

def field(shape, bc):
    """A near-constant background (the MSD wall's use) with smooth structure that vanishes at walls."""
    y, x = np.meshgrid(*[np.arange(n) / n for n in shape], indexing="ij")
    r = 0.05 * np.sin(2 * np.pi * (x + 2 * y) + 0.4) * (1.0 if bc == "periodic" else np.sin(np.pi * x) * np.sin(np.pi * y))
    return (1.0 + r) * np.exp(0.1j * np.cos(np.pi * (x - y)))


SHAPES = [(3, 3), (3, 40), (4, 5), (16, 17), (33, 65), (50, 131), (97, 64)]


def run(psi, V, bc, order, dtype, variant, tile, steps):
    h, a, s = 0.3, 0.7, -1.0
    dt = 0.2 * max_dt(2, h, a, order, 0.0 if V is None else float(np.max(np.abs(V))), 2.0)
    g = Integrator(psi, h, a, s, V, bc, order, dtype)
    g.set_kernel(variant, tile)
    for n in steps:
        g.step(n, dt)
    g.sync()
    out = g.numpy()
    g.close()
    return out


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dtype", ["c128", "c64", "c64_acc64"])
def test_whole_step_equals_per_site_bitwise(shape, bc, order, dtype):
    psi = field(shape, bc)
    for V in (None, W.random_potential(shape, 5, 0.1)):
        for steps in ((1,), (2, 19)):
            ref = run(psi, V, bc, order, dtype, 0, -1, steps)
            for tile in (-1, 0, 1, 2, 3):
                assert np.array_equal(run(psi, V, bc, order, dtype, 1, tile, steps), ref), (tile, steps, V is None)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("order", [2, 4])
def test_whole_fp64_step_equals_per_site_exact_sum_bitwise(shape, bc, order):
    """The FP64 whole step (exact-sum stencil) against the one-thread-per-site exact-sum kernel."""
    psi = field(shape, bc)
    for V in (None, W.random_potential(shape, 5, 0.1)):
        for steps in ((1,), (2, 19), (5,)):
            ref = run(psi, V, bc, order, "c128", 3, -1, steps)
            assert np.array_equal(run(psi, V, bc, order, "c128", 2, -1, steps), ref), (steps, V is None)
