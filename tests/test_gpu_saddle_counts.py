"""Operator applications of the velocity-pressure solve with a long basis and a tight tolerance, at the larger density ratio: no
more than one classical Gram-Schmidt pass with the DGKS threshold 1/2 and a checked inner solve take (15, 15, 20 and 20 of
them), but for what the FP32 atomics of the inner solve move from run to run."""
import numpy as np
import pytest

import workloads
from oracle import momentum
from test_gpu_parity import cuda, make_op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,newton,most", [(3, 0, 15), (3, 1, 15), (2, 0, 20), (2, 1, 20)])
def test_applications(p, newton, most):
    n = 12
    wl = workloads.random_workload(n, p, 90 + n, geom="deformed", ratio=1e4, dirichlet_faces=0x1F, newton=newton)
    f = np.random.default_rng(n).uniform(-1, 1, 3 * (p * n + 1) ** 3)
    f[momentum.Problem.from_workload(wl).constrained()] = 0.0
    _, _, info = make_op(wl).solve_saddle(cuda(f), rtol=1e-12, restart=200)
    assert info["converged"] and info["iters"] <= most + 2, info
