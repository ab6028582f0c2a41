"""The accuracy of the momentum apply against FP64, as the geometric mean over a fixed set of small cases: coefficients rounded
once to a pair, line sums normalized before they are multiplied or added twice, FP32 sums of values and tests paired.

Bars: the means of the kernels that formed every product and sum point by point with Q-term dot products (2 % more: the
means' repeatability is a few tenths of a per cent, from the order of the atomic adds).
"""
import numpy as np
import pytest

import workloads
from oracle import momentum
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
