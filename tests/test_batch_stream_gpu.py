"""The batch reads its runs' V and Psi in stream order: a device kernel that rewrites them right before a call is seen by
that call's first step, whether it is launched by itself or heads a graph."""
import numpy as np
import pytest
import torch

from paper_1203_1263_gb300 import workloads as W
from paper_1203_1263_gb300.integrator import BatchIntegrator, max_dt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps", [1, 2, 3, 16, 19])
def test_potential_written_on_the_stream_right_before_a_call(steps):
    runs = []
    for i, shape in enumerate([(70, 90), (64, 64), (33, 120)]):
        runs.append(dict(psi0=np.ones(shape) * np.exp(0.1j * i), h=0.3, a=0.7, s=-1.0, V=W.random_potential(shape, 5 + i, 0.1),
                         dt=0.2 * max_dt(2, 0.3, 0.7, 4, 2.0, 2.0), bc=("dirichlet", "msd", "l0")[i], order=(4, 2, 4)[i]))
    big = torch.ones(1 << 26, device="cuda")
    out = []
    for wait in (True, False):
        b = BatchIntegrator(runs)
        for k in range(4):
            big.mul_(1.0)   # keeps the stream busy while the host goes on
            for i, (v, p) in enumerate(zip(b.V, b.psi)):
                v.copy_(torch.as_tensor(runs[i]["V"], dtype=torch.float32), non_blocking=False)
                v.mul_(1.0 + 3.0 * k)
                p.mul_(complex(0.8, 0.6))
            if wait:
                torch.cuda.synchronize()
            b.step(steps)
        b.sync()
        out.append([b.numpy(i) for i in range(len(runs))])
        b.close()
    assert all(np.array_equal(x, y) for x, y in zip(*out))
