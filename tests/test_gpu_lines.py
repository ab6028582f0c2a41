"""The line-sweep kernels (FP64-accurate and FP32 momentum apply, adjoint) where their cell groups end: one cell, fewer
cells than a group, a last group that is partly filled, rows that run on inside a group; every face open or closed."""
import numpy as np
import pytest

import workloads
from oracle import adjoint, momentum
from test_gpu_parity import cuda, make_op, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("faces", [0, 0x3F, 0x1A])
@pytest.mark.parametrize("n,p", [(1, 2), (1, 3), (3, 2), (5, 3), (7, 2)])
def test_cell_groups(n, p, faces):
    wl = workloads.random_workload(n, p=p, seed=3 * n + p, geom="deformed", dirichlet_faces=faces)
    op = make_op(wl)
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
    assert rel(g["x"], adjoint.grad_x(pb, w, wp)) <= 1e-12
    for k, want in (("u0", gu), ("phi", gphi), ("mdot", gm)):
        assert rel(g[k], want) <= 1e-12 or np.linalg.norm(want) == 0.0
