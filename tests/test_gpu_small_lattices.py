"""The single-launch solvers, the quadrature-point cache and the surface force where their index ranges end: lattices of one
to three cells (every stencil row meets the boundary, fewer nodes than a block has threads), cell counts that are no
multiple of a block's cells, a level set whose far field holds a NaN.  Bars as in the tests of the same entry points at
ordinary sizes: level-set solves 1e-10 (1e-9 after two pseudo-steps), saddle solves 1e-7 and 1e-6, Jacobi diagonal 2e-5."""
import numpy as np
import pytest

import workloads
from oracle import fe, geometry, momentum, saddle, solve
from test_gpu_parity import cuda, make_op, rel

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore::scipy.sparse.SparseEfficiencyWarning")]


@pytest.mark.parametrize("n", [1, 2, 3])
def test_level_set_solves(n):
    wl = workloads.random_workload(n, 2, 30 + n, geom="sphere")
    wl.phi = np.random.default_rng(n).uniform(-0.9, 0.9, (n + 1) ** 3)
    op = make_op(wl)
    mesh = fe.Mesh(n, 1, wl.L)
    nf, info = op.projected_normal()
    ref = geometry.projected_normal(mesh, wl.phi, wl.params["eta_n"])
    assert info["converged"] and rel(nf, ref.ravel()) < 1e-10
    kappa, info = op.curvature(cuda(ref.ravel()))
    assert info["converged"] and rel(kappa, geometry.curvature(mesh, ref, wl.params["eta_kappa"])) < 1e-10
    op.set_levelset_normal(cuda(ref.ravel()))
    psi, info = op.reinitialize(cuda(wl.phi), 2)
    want, _ = geometry.reinitialize(mesh, wl.phi, ref, wl.params["eps"], wl.params["dtau"], 2, psi0=wl.phi)
    assert info["converged"] and rel(psi, want) < 1e-9


@pytest.mark.parametrize("n,p,faces", [(3, 2, 0x0F), (1, 3, 0x1F)])
def test_saddle_solve(n, p, faces):
    wl = workloads.random_workload(n, p, 40 + n, geom="sphere", dirichlet_faces=faces)
    op = make_op(wl)
    pb = momentum.Problem.from_workload(wl)
    f = np.random.default_rng(n + p).uniform(-1, 1, 3 * op.n_u)
    f[pb.constrained()] = 0.0
    x, pr, info = op.solve_saddle(cuda(f), rtol=1e-12, max_iter=2000)
    xr, prr = saddle.solve(pb, f)
    assert info["converged"], info
    assert rel(x, xr) < 1e-7 and rel(pr, prr) < 1e-6


@pytest.mark.parametrize("n,p", [(1, 2), (3, 2), (5, 2), (1, 3), (3, 3)])
def test_jacobi_diagonal_of_the_last_cells(n, p):
    wl = workloads.random_workload(n, p, 50 + n, geom="deformed", dirichlet_faces=0)
    d = make_op(wl).jacobi_diagonal().cpu().numpy()
    np.testing.assert_allclose(d, solve.jacobi_diagonal(momentum.Problem.from_workload(wl)), rtol=2e-5)


def test_surface_force_keeps_a_nan_of_the_far_field():
    """A NaN curvature at a corner node, where the interface delta vanishes: NaN on the nodes of that node's cell (0 times
    NaN), the other entries as without it."""
    n, p = 8, 2
    wl = workloads.random_workload(n, p, 3, geom="sphere", dirichlet_faces=0)
    op = make_op(wl)
    nf, _ = op.projected_normal()
    kappa, _ = op.curvature(nf)
    want = op.surface_tension(nf, kappa, 1.0).cpu().numpy()
    kappa[0] = float("nan")
    got = op.surface_tension(nf, kappa, 1.0).cpu().numpy()
    m = p * n + 1
    hit = np.zeros((3, m, m, m), bool)
    hit[:, : p + 1, : p + 1, : p + 1] = True
    hit = hit.ravel()
    assert np.isnan(got[hit]).all() and np.abs(got[~hit] - want[~hit]).max() <= 1e-14 * np.abs(want).max()
