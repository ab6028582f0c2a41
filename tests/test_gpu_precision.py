"""The accuracy of the momentum applies and the adjoint against FP64, as the geometric mean over a fixed set of small cases:
coefficients rounded once to a pair, line sums normalized before they are multiplied or added twice, FP32 sums of values and
tests paired.

Bars: the means of the kernels that formed every product and sum point by point with Q-term dot products (2 % more: the
means' repeatability is a few tenths of a per cent, from the order of the atomic adds).
"""
import numpy as np
import pytest
import torch

import workloads
from oracle import adjoint, fe, levelset, momentum
from test_gpu_parity import cuda, make_op, rel

pytestmark = pytest.mark.gpu


def mean_errors(p, prec):
    """Geometric means of the relative errors of y and y_p."""
    e = []
    for k in range(24):
        wl = workloads.random_workload(4 + k % 4, p, 500 + k, geom=("sphere", "deformed", "slab")[k % 3],
                                       dirichlet_faces=(0x3F, 0x1F)[k % 2])
        x = wl.x.astype(np.float32) if prec == 32 else wl.x
        y, yp = make_op(wl).apply_momentum(cuda(x), prec=prec, with_divergence=True)
        yo, ypo = momentum.apply(momentum.Problem.from_workload(wl), x.astype(np.float64), with_divergence=True)
        e.append((rel(y.double(), yo), rel(yp.double(), ypo)))
    return np.exp(np.log(np.array(e)).mean(0))


BARS = {(2, 64): (5.447e-15, 5.549e-15), (3, 64): (8.696e-15, 1.0628e-14), (2, 32): (1.447e-7, 1.96e-7),
        (3, 32): (1.3507e-7, 1.535e-7)}


@pytest.mark.parametrize("p,prec", sorted(BARS))
def test_mean_error(p, prec):
    got, bar = mean_errors(p, prec), BARS[p, prec]
    print(f"mean errors Q{p} FP{prec}: {got[0]:.3e} {got[1]:.3e}")
    assert got[0] <= 1.02 * bar[0] and got[1] <= 1.02 * bar[1]


def mean_pressure_error(p):
    """Of the pressure term alone: the velocity rows of the velocity-pressure apply at x = 0, and the oracle's -B^T p."""
    e = []
    for k in range(12):
        wl = workloads.random_workload(3 + k % 3, p, 600 + k, geom="sphere", dirichlet_faces=0x1F)
        op = make_op(wl)
        pr = np.random.default_rng(k).uniform(-1, 1, op.n_p)
        y, _ = op.apply_saddle(torch.zeros(3 * op.n_u, dtype=torch.float64, device="cuda"), cuda(pr))
        B, _ = momentum.divergence(momentum.Problem.from_workload(wl))
        e.append(rel(y, -(B.T @ pr)))
    return np.exp(np.log(e).mean())


def mean_adjoint_errors(p):
    """Of g_x, g_u0 and g_phi."""
    e = []
    for k in range(60):
        wl = workloads.random_workload(4, p, 700 + k, geom=("sphere", "deformed", "slab")[k % 3])
        pb = momentum.Problem.from_workload(wl)
        rng = np.random.default_rng(k)
        w, wp = rng.uniform(-1, 1, wl.x.shape), rng.uniform(-1, 1, 5 ** 3)
        g = make_op(wl).apply_adjoint(cuda(w), cuda(wl.x), cuda(wp))
        gu, gphi, _ = adjoint.param_gradients(pb, wl.x, w, wp)
        e.append((rel(g["x"], adjoint.grad_x(pb, w, wp)), rel(g["u0"], gu), rel(g["phi"], gphi)))
    return np.exp(np.log(np.array(e)).mean(0))


def test_mean_error_of_the_pressure_term():
    got = mean_pressure_error(2)
    print(f"mean error, pressure term: {got:.3e}")
    assert got <= 1.02 * 5.484e-15


def test_mean_errors_of_the_adjoint():
    got = mean_adjoint_errors(2)
    print("mean errors, adjoint:", got)
    assert (got <= 1.02 * np.array([4.702e-15, 8.542e-15, 4.686e-15])).all()


def mean_levelset_errors():
    """Of the FP32 level-set operators: reinitialization, its explicit side, advection."""
    e = []
    for k in range(40):
        n = 3 + k % 6
        wl = workloads.random_workload(n, 2, 800 + k, geom=("sphere", "deformed", "slab")[k % 3])
        op, mesh, rng = make_op(wl), fe.Mesh(n, 2, 1.0), np.random.default_rng(k)
        ug = rng.uniform(-1, 1, 3 * mesh.n_phi)
        op.set_transport_velocity(cuda(ug))
        x = rng.uniform(-1, 1, mesh.n_phi).astype(np.float32)
        e.append([rel(op.apply_levelset(cuda(x), mode=m, prec=32).double(),
                      levelset.apply(mesh, m, x.astype(np.float64), wl.phi, ug, wl.params))
                  for m in ("reinit", "reinit_rhs", "advect")])
    return np.exp(np.log(np.array(e)).mean(0))


def test_mean_errors_of_the_fp32_levelset_operators():
    got = mean_levelset_errors()
    print("mean errors, FP32 level set:", got)
    assert (got <= 1.02 * np.array([6.87e-8, 7.05e-8, 8.04e-8])).all()
