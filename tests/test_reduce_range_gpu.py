"""Sums that leave the FP64 range while every term is finite: the result is not finite, as with sums in FP64 (never the
sum of the blocks that stayed in range).  The sums overflow inside one block, inside every block, or only when the
blocks are added."""
import math

import numpy as np
import pytest
import torch

from paper_1203_1263_gb300 import _lib as L
from paper_1203_1263_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
BIG = 1.2e154   # BIG^2 = 1.44e308: one term is in range, two are not


@pytest.mark.parametrize("n,at", [(3, (0, 2)), (257, (0, 256)), (5000, (1, 100)), (5000, (17, 4000)), (300001, slice(None))])
@pytest.mark.parametrize("dtype", ["c128", "c64_acc64"])
def test_an_overflowing_mass_is_not_finite(n, at, dtype):
    psi = np.ones(n, complex)
    psi[at if isinstance(at, slice) else list(at)] = BIG
    g = Integrator(psi, 0.25, 0.7, 0.0, None, "dirichlet", 2, dtype)
    assert not math.isfinite(g.mass())
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    code = {"c128": L.C128, "c64_acc64": L.C64_ACC64}[dtype]
    L.check(L.lib().nlse_mass_noalloc(1, L.int64_array((n,)), 0.25, code, g.psi.data_ptr(), out.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream))
    assert not math.isfinite(float(out.item()))
    g.psi.fill_(0.5)
    assert abs(g.mass() - 0.25 * 0.25 * n) <= 1e-13 * n   # the next reduction is not affected


@pytest.mark.parametrize("shape", [(257,), (60, 70), (11, 20, 30)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_an_overflowing_energy_is_not_finite(shape, bc):
    # V |Psi|^2 = 0.6e308 at each interior site; |Psi|^4 and a |Psi Lap Psi| stay in range
    g = Integrator(np.full(shape, 1e74, complex), 1.0, 1e160, 0.0, np.full(shape, 0.6e160), bc, 4, "c128")
    assert not math.isfinite(g.energy())
