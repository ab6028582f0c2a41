"""The surface force with a factor that is not finite: 0 times it is NaN, also in the cells where the interface delta
vanishes (Eq. surfaceTension: every quadrature point carries alpha kappa n delta rho)."""
import numpy as np
import pytest
import torch

import workloads
from test_gpu_parity import cuda, make_op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,n_sub", [(8, 2, 1), (10, 3, 2)])
@pytest.mark.parametrize("alpha", [float("nan"), float("inf")])
def test_alpha_not_finite(n, p, n_sub, alpha):
    wl = workloads.random_workload(n, p, 3, geom="sphere", dirichlet_faces=0, n_sub=n_sub)
    op = make_op(wl)
    nf = torch.ones(3 * op.n_phi, dtype=torch.float64, device="cuda")  # a direction at every point
    kappa = torch.full((op.n_phi,), 2.0, dtype=torch.float64, device="cuda")
    f = op.surface_tension(nf, kappa, alpha).cpu().numpy().reshape(3, p * n + 1, p * n + 1, p * n + 1)
    assert np.isnan(f[:, : p + 1, : p + 1, : p + 1]).all()  # a corner cell, far from the interface
    if np.isnan(alpha):
        assert np.isnan(f).all()


def test_curvature_that_overflows_with_alpha():
    n, p = 8, 2
    op = make_op(workloads.random_workload(n, p, 3, geom="sphere", dirichlet_faces=0))
    nf = torch.ones(3 * op.n_phi, dtype=torch.float64, device="cuda")
    kappa = torch.full((op.n_phi,), 1e200, dtype=torch.float64, device="cuda")
    f = op.surface_tension(nf, kappa, 1e200).cpu().numpy().reshape(3, p * n + 1, p * n + 1, p * n + 1)
    assert np.isnan(f[:, : p + 1, : p + 1, : p + 1]).all()
