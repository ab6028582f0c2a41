"""Edges that the neighbouring files leave out: the single-launch solvers on subdivided level-set meshes of one to three velocity
cells, and the deterministic line kernels where a group of cells is partly filled and faces are open.  Bars as in those files."""
import numpy as np
import pytest

import workloads
from oracle import adjoint, fe, geometry, momentum
from test_gpu_parity import cuda, make_op, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3])
def test_level_set_solves_subdivided(n):
    wl = workloads.random_workload(n, 2, 30 + n, geom="sphere", n_sub=2)
    wl.phi = np.random.default_rng(n).uniform(-0.9, 0.9, (2 * n + 1) ** 3)
    op = make_op(wl)
    mesh = fe.Mesh(2 * n, 1, wl.L)
    nf, info = op.projected_normal()
    ref = geometry.projected_normal(mesh, wl.phi, wl.params["eta_n"])
    assert info["converged"] and rel(nf, ref.ravel()) < 1e-10
    kappa, info = op.curvature(cuda(ref.ravel()))
    assert info["converged"] and rel(kappa, geometry.curvature(mesh, ref, wl.params["eta_kappa"])) < 1e-10
    op.set_levelset_normal(cuda(ref.ravel()))
    psi, info = op.reinitialize(cuda(wl.phi), 2)
    want, _ = geometry.reinitialize(mesh, wl.phi, ref, wl.params["eps"], wl.params["dtau"], 2, psi0=wl.phi)
    assert info["converged"] and rel(psi, want) < 1e-9


@pytest.mark.parametrize("n,p,faces", [(1, 2, 0), (3, 2, 0x1A), (5, 2, 0), (3, 3, 0), (5, 3, 0x1A)])
def test_deterministic_cell_groups(n, p, faces):
    wl = workloads.random_workload(n, p=p, seed=5 * n + p, geom="deformed", dirichlet_faces=faces)
    op = make_op(wl)
    op.set_deterministic(True)
    pb = momentum.Problem.from_workload(wl)
    y, yp = op.apply_momentum(cuda(wl.x), prec=64, with_divergence=True)
    yo, ypo = momentum.apply(pb, wl.x, with_divergence=True)
    assert rel(y, yo) <= 1e-12 and rel(yp, ypo) <= 1e-12
    x32 = wl.x.astype(np.float32)
    y, yp = op.apply_momentum(cuda(x32), prec=32, with_divergence=True)
    yo, ypo = momentum.apply(pb, x32.astype(np.float64), with_divergence=True)
    assert rel(y.double(), yo) <= 2e-5 and rel(yp.double(), ypo) <= 2e-5
    rng = np.random.default_rng(n)
    w, wp = rng.uniform(-1, 1, wl.x.shape), rng.uniform(-1, 1, (n + 1) ** 3)
    g = op.apply_adjoint(cuda(w), cuda(wl.x), cuda(wp))
    gu, gphi, gm = adjoint.param_gradients(pb, wl.x, w, wp)
    for k, want in (("x", adjoint.grad_x(pb, w, wp)), ("u0", gu), ("phi", gphi), ("mdot", gm)):
        assert np.linalg.norm(want) > 0.0 and rel(g[k], want) <= 1e-12, k
