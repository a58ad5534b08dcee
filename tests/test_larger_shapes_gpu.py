"""Branches of the dispatch that only larger or longer grids enter, each bit for bit against one thread per site: the
whole-step FP64 kernel's 16-row tiles, the FP32 columns in one wave and with odd rows above three million sites, the
FP32 TMA tiles with their wall slabs or shells at ragged sizes, long FP32 lines, and FP64 grids of up to 600,000 sites
with a lane per component."""
import numpy as np
import pytest
import torch

from paper_1203_1263_gb300.integrator import Integrator, max_dt

pytestmark = pytest.mark.gpu


def state(shape, bc):
    g = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float64) / n for n in shape], indexing="ij")
    r = 0.05 * torch.sin(2 * np.pi * (sum((k + 1) * x for k, x in enumerate(g))) + 0.4)
    if bc != "periodic":
        for x in g:
            r = r * torch.sin(np.pi * x)
    psi = (1.0 + r) * torch.exp(0.1j * torch.cos(2 * np.pi * (g[0] - g[-1])))
    return psi, 0.1 * sum(torch.cos(9.0 * x) for x in g)


def same(shape, bc, order, dtype, ref, variants, steps=(3, 16), with_v=True):
    psi, V = state(shape, bc)
    dt = 0.2 * max_dt(len(shape), 0.3, 0.7, order, 0.3, 2.0)
    out = None
    for variant, tile in [(ref, -1)] + list(variants):
        g = Integrator(psi, 0.3, 0.7, -1.0, V if with_v else None, bc, order, dtype)
        if variant is not None:
            g.set_kernel(variant, tile)
        for n in steps:
            g.step(n, dt)
        g.sync()
        if out is None:
            out = g.psi.clone()
            assert torch.isfinite(torch.view_as_real(out)).all()
        else:
            assert torch.equal(g.psi, out), (variant, tile)
        g.close()


@pytest.mark.parametrize("shape", [(256, 256), (201, 255), (273, 270), (17, 4500)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("order", [2, 4])
def test_whole_fp64_step_on_16_row_tiles(shape, bc, order):
    same(shape, bc, order, "c128", 3, [(2, -1)])


@pytest.mark.parametrize("shape,dtypes", [((103, 107, 109), ("c64_acc64",)), ((141, 149, 151), ("c64", "c64_acc64"))])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0"])
@pytest.mark.parametrize("order", [2, 4])
def test_columns_of_large_grids(shape, dtypes, bc, order):
    for dtype in dtypes:
        same(shape, bc, order, dtype, 0, [(1, -1)])


@pytest.mark.parametrize("shape", [(150, 142, 148), (7, 690, 650), (620, 9, 560), (560, 554, 10), (6, 720, 710), (590, 880, 6)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0"])
@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64"])
def test_fp32_tma_tiles_and_walls_at_ragged_sizes(shape, bc, order, dtype):
    assert shape[0] * shape[1] * shape[2] > 3000000
    same(shape, bc, order, dtype, 0, [(1, t) for t in range(4)], steps=(3,))


@pytest.mark.parametrize("shape", [(6, 600, 700), (3, 300, 400), (300, 5, 300)])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64", "c128"])
@pytest.mark.parametrize("order", [2, 4])
def test_flat_grids_of_msd_walls(shape, dtype, order):
    same(shape, "msd", order, dtype, 0, [(1, -1)], steps=(3,))
    if dtype == "c128":
        same(shape, "msd", order, dtype, 3, [(2, -1)], steps=(3,))


@pytest.mark.parametrize("n", [200001, 250003])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0", "periodic"])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64"])
def test_long_fp32_lines(n, bc, dtype):
    for order in (2, 4):
        same((n,), bc, order, dtype, 0, [(1, -1)], steps=(1, 19))


@pytest.mark.parametrize("shape", [(41, 37, 43), (80, 75, 70)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0"])
@pytest.mark.parametrize("order", [2, 4])
def test_a_lane_per_component_on_larger_grids(shape, bc, order):
    same(shape, bc, order, "c128", 0, [(1, -1)], steps=(3,))


@pytest.mark.parametrize("shape", [(5, 6000), (3, 20000), (12, 5000), (6, 30000), (128, 128), (100, 700), (500, 420)])
@pytest.mark.parametrize("bc", ["dirichlet", "msd", "l0"])
@pytest.mark.parametrize("order", [2, 4])
def test_fp64_planes_with_either_form_of_the_walls(shape, bc, order):
    same(shape, bc, order, "c128", 0, [(1, -1), (None, -1)][:2 if shape[0] * shape[1] <= 80000 and shape != (128, 128) else 1],
         steps=(5,))
    same(shape, bc, order, "c128", 3, [(2, -1)], steps=(5,))
