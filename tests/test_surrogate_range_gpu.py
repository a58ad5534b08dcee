"""Non-finite states through the surrogate's sums: an infinite term makes the loss and the states' masses infinite and
a NaN makes them NaN, as sums in FP64 do; the batch's other states keep their masses."""
import math

import numpy as np
import pytest
import torch

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.surrogate import Surrogate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [math.inf, -math.inf, math.nan])
@pytest.mark.parametrize("site", [0, 24 * 28 - 1])
def test_masses_and_loss_with_a_non_finite_term(bad, site):
    H, Wd, nb = 24, 28, 3
    sur = Surrogate(H, Wd, channels=16, layers=3, dilations=(1, 2, 1), max_batch=nb, seed=3)
    psi = torch.as_tensor(W.random_field((nb, H, Wd), 4), dtype=torch.complex64).cuda()
    target = psi.clone()
    target.view(nb, -1)[1, site] = complex(0.25, bad)
    _, loss = sur.gradients(psi, target)
    assert math.isnan(loss) if math.isnan(bad) else loss == math.inf
    masses = torch.zeros((nb, 2), dtype=torch.float64, device="cuda")
    ref = torch.zeros((nb, 2), dtype=torch.float64, device="cuda")
    sur.forward(psi, masses=ref)
    sur.forward(target, masses=masses)
    m, r = masses.cpu().numpy(), ref.cpu().numpy()
    assert np.isnan(m[1, 0]) if math.isnan(bad) else m[1, 0] == math.inf
    assert np.array_equal(m[[0, 2]], r[[0, 2]]) and np.all(np.isfinite(r))
