"""nlse_autotune on FP32 3D grids whose steps take the columns kernel, which no tile shape changes: the default (or the
caller's) tile is kept, however the timings fall, and the tune file never gets another."""
import numpy as np
import pytest

from paper_1203_1263_gb300.integrator import Integrator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,default", [((12, 30, 72), 0), ((9, 31, 71), 0), ((11, 90, 96), 3)])
@pytest.mark.parametrize("dtype", ["c64", "c64_acc64"])
@pytest.mark.parametrize("chosen", [-1, 2])
def test_the_default_tile_is_kept(shape, default, dtype, chosen, tmp_path, monkeypatch):
    monkeypatch.setenv("NLSE_TUNE_CACHE", str(tmp_path / "tune.txt"))
    # a potential keeps the two choices' cache entries apart
    V = np.full(shape, 0.1) if chosen == 2 else None
    g = Integrator(np.ones(shape, complex), 0.3, 0.7, -1.0, V, "msd", 4, dtype)
    g.set_kernel(1, chosen)
    cfg, ms = g.autotune()
    want = chosen if chosen >= 0 else default
    assert cfg == want and ms > 0
    lines = (tmp_path / "tune.txt").read_text().splitlines()
    assert len(lines) == 1 and lines[0].endswith(f"={want}")
