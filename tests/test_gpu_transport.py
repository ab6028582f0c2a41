"""Closest-point pass on short band lists: fewer band nodes than the pass has lanes, so that several lanes project the
trial points of one node from the start or soon after it (App. C)."""
import numpy as np
import pytest

import workloads
from oracle import fe, physics, transport
from test_gpu_parity import make_op

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,variant,geom,n_sub", [(1, 2, 2, "slab", 1), (2, 2, 3, "slab", 1), (5, 2, 2, "sphere", 1),
                                                    (7, 3, 3, "deformed", 1), (4, 3, 2, "sphere", 2),
                                                    (9, 2, 2, "deformed", 1)])
def test_short_band_lists(n, p, variant, geom, n_sub):
    """u_Gamma is the variant's formula at the point the pass returns (to rounding), and an unflagged point lies on the
    isocontour to 1e-8 h (the projection stops at 1e-10 h)."""
    wl = workloads.random_workload(n, p=p, seed=11, geom=geom, variant=variant, eps=0.3 / n, n_sub=n_sub)
    op = make_op(wl)
    ug, flags, nflag = op.transport_velocity()
    ug, flags = ug.cpu().numpy().reshape(3, -1), flags.cpu().numpy()
    assert nflag == int(flags.sum())
    mesh = fe.Mesh(n, p, 1.0, n_sub)
    eps, h, m1 = wl.params["eps"], mesh.h / n_sub, n * n_sub + 1
    d_t, rho_t = (3.0 * eps, wl.params["rho_l"]) if variant == 2 else (-3.0 * eps, wl.params["rho_g"])
    lo, hi = (-physics.PHI_GAS_BAND, physics.PHI_BAND) if variant == 2 else (-physics.PHI_BAND, physics.PHI_GAS_BAND)
    y = op.closest_points().cpu().numpy() / h
    ev = transport.PointEval(mesh, wl.phi, wl.u0)
    for k in range(op.n_phi):
        x = np.array([k % m1, (k // m1) % m1, k // (m1 * m1)], dtype=float)
        band = lo < wl.phi[k] < hi
        assert band or (flags[k] == 0 and np.array_equal(y[:, k] * h, x * h))
        expect = ev.velocity(y[:, k]) + wl.mdot[k] / rho_t * physics.normal(ev.phi_grad(x)[1], h)
        assert np.abs(ug[:, k] - expect).max() <= 1e-12 * np.abs(ug).max()
        if band and flags[k] == 0:
            assert abs(float(physics.distance(ev.phi_grad(y[:, k])[0], eps)) - d_t) <= 1e-8 * h
