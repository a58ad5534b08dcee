"""Mass sums on states whose terms span many magnitudes, signs and block shares: the integer sums are exact,
so the result is the correctly rounded sum up to the final pair additions (a few units of 2^-53)."""
import math

import numpy as np
import pytest
import torch

from paper_1203_1263_gb300 import _lib as L
from paper_1203_1263_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu
CODES = {"c128": L.C128, "c64": L.C64, "c64_acc64": L.C64_ACC64}


def state(n, dtype, kind):
    rng = np.random.default_rng(n)
    span = 15 if dtype == "c64" else 120
    if kind == "rising":      # every term raises the running exponent
        mag = np.linspace(-span, span, n)
    elif kind == "falling":
        mag = np.linspace(span, -span, n)
    else:
        mag = rng.uniform(-span, span, n)
    z = 10.0 ** mag * np.exp(2j * np.pi * rng.random(n))
    z[n // 2] = 0.0
    return z.astype(np.complex64 if dtype == "c64" else np.complex128)


@pytest.mark.parametrize("n", [3, 255, 257, 4096, 300001])
@pytest.mark.parametrize("kind", ["rising", "falling", "random"])
@pytest.mark.parametrize("dtype", ["c128", "c64", "c64_acc64"])
def test_mass_sums_are_exact(n, kind, dtype):
    z = state(n, dtype, kind)
    x = np.concatenate([z.real, z.imag]).astype(np.float64)
    ref = 0.25 * math.fsum(x * x)
    g = Integrator(z, 0.25, 0.7, -1.0, None, "dirichlet", 2, dtype)
    assert abs(g.mass() - ref) <= 8 * 2.0 ** -53 * ref
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    L.check(L.lib().nlse_mass_noalloc(1, L.int64_array((n,)), 0.25, CODES[dtype], g.psi.data_ptr(), out.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream))
    assert abs(float(out.item()) - ref) <= 8 * 2.0 ** -53 * ref


@pytest.mark.parametrize("dtype", ["c128", "c64", "c64_acc64"])
@pytest.mark.parametrize("bad", [math.nan, math.inf])
def test_a_non_finite_term_shows(dtype, bad):
    z = state(5000, dtype, "random")
    g = Integrator(z, 0.25, 0.7, -1.0, None, "dirichlet", 2, dtype)
    g.psi[4321] = complex(0.0, bad)
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    L.check(L.lib().nlse_mass_noalloc(1, L.int64_array((5000,)), 0.25, CODES[dtype], g.psi.data_ptr(), out.data_ptr(),
                                      torch.cuda.current_stream().cuda_stream))
    assert not math.isfinite(float(out.item()))
    for call in (g.mass, g.energy):
        with pytest.raises(L.NLSEError) as e:
            call()
        assert e.value.code == L.NLSE_ENONFINITE
