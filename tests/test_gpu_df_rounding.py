"""Rounding error of the float-float product of two SU(3) matrices, as the FP32
link update multiplies its exponential onto the links, against extended precision:
no more than with products of twelve instructions and one error sum, whose root
mean square errors for these inputs are the bounds (half a percent added).  The
exponential is what the update makes of unit links; the links come from an earlier
update, so both are float-float numbers already."""
import numpy as np
import pytest

from paper_1212_0785_gb300 import lqcd

pytestmark = pytest.mark.gpu

DIMS, V = (8, 8, 8, 8), 4096
BOUND = {0.1: 1.964e-15, 0.5: 2.066e-15, 4.0: 2.093e-15}


def update(U, P, c):
    G = lqcd.gauge_field(DIMS).upload(U)
    lqcd.link_update(G, P, c, arith=lqcd.F32)
    return G.download()


def test_link_product():
    r = np.random.default_rng(11)
    one = np.broadcast_to(np.eye(3), (V, 4, 3, 3)).astype(complex)
    for c, bound in BOUND.items():
        P, Q = (lqcd.momentum_field(DIMS).upload(r.standard_normal((V, 4, 8))) for _ in range(2))
        U, E = update(one, Q, 4.0), update(one, P, c)
        a, b = E.astype(np.clongdouble), U.astype(np.clongdouble)
        ref = sum(a[..., :, k, None] * b[..., k, None, :] for k in range(3))
        err = float(np.sqrt((np.abs(update(U, P, c) - ref) ** 2).mean()))
        assert err <= 1.005 * bound, (c, err, bound)
