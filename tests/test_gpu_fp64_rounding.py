"""Rounding errors of the FP64 kernels against extended precision: the root mean
square error of each result may not exceed that of the plain order of operations,
in which a sum of complex products rounds each product and then the sum, and the
exponential takes its angles from arccos, sin and cos.  The bounds are that
order's errors (fused multiply-adds where the compiler contracts), measured for
these inputs; half a percent is added for inputs that another LAPACK rounds
differently."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1212_0785_gb300 import lqcd
from tests.gpu_util import full_from_half
from tests.lattice_np import shift

pytestmark = pytest.mark.gpu

DIMS, V = (8, 8, 8, 8), 4096
L, C = np.longdouble, np.clongdouble
BOUND = {"hop": 1.447e-16, "hop_dag": 1.464e-16, "gauge_force": 1.844e-16, "row1": 6.22e-17, "row2": 8.36e-17,
         0.02: 1.543e-16, 0.1: 1.572e-16, 0.4: 1.709e-16, 0.7: 1.951e-16, 1.0: 2.322e-16, 4.0: 6.706e-16,
         "plaquette": 5.584e-16}


def mm(a, b):
    return sum(a[..., :, k, None] * b[..., k, None, :] for k in range(3))


def dag(a):
    return np.conj(np.swapaxes(a, -1, -2))


def rand_su3(r, n):
    a = r.standard_normal((n, 3, 3)) + 1j * r.standard_normal((n, 3, 3))
    q, _ = np.linalg.qr(a)
    q[:, 2] = np.conj(np.cross(q[:, 0], q[:, 1]))
    return q


def rms(err, ref=None):
    e = np.sqrt((np.abs(err) ** 2).mean())
    return float(e if ref is None else e / np.sqrt((np.abs(ref) ** 2).mean()))


def check(name, value):
    assert value <= 1.005 * BOUND[name], (name, value, BOUND[name])


@pytest.fixture(scope="module")
def inputs():
    r = np.random.default_rng(5)
    U = rand_su3(r, V * 4).reshape(V, 4, 3, 3)
    psi = r.standard_normal((V // 2, 4, 3)) + 1j * r.standard_normal((V // 2, 4, 3))
    return U, psi, r.standard_normal((V, 4, 8))


def gammas():
    g = np.zeros((4, 4, 4), C)
    for mu, rows in enumerate([((3, 1j), (2, 1j), (1, -1j), (0, -1j)), ((3, -1), (2, 1), (1, 1), (0, -1)),
                               ((2, 1j), (3, -1j), (0, -1j), (1, 1j)), ((2, 1), (3, 1), (0, 1), (1, 1))]):
        for a, (c, v) in enumerate(rows):
            g[mu, a, c] = v
    return g


@pytest.mark.parametrize("name", ["hop", "hop_dag"])
def test_hop(inputs, name):
    U, psi, _ = inputs
    out = lqcd.spinor_field(DIMS, 1)
    lqcd.dslash(out, lqcd.gauge_field(DIMS).upload(U), lqcd.spinor_field(DIMS, 0).upload(psi), name == "hop_dag")
    p, u, f = full_from_half(psi, DIMS, 0).astype(C), U.astype(C), 1 if name == "hop_dag" else -1
    ref, t, last = np.zeros((V, 4, 3), C), np.arange(V) // 512, DIMS[3] - 1
    for mu, g in enumerate(gammas()):
        g = np.array([[1 if i == j else 0 for j in range(4)] for i in range(4)], C) + f * g
        h = shift(sum(g[:, s, None] * p[:, None, s] for s in range(4)), DIMS, mu, 1)
        h[(t == last) & (mu == 3)] *= -1
        ref += sum(u[:, mu, None, :, b] * h[:, :, b, None] for b in range(3))
        g = 2 * np.eye(4) - g
        h = sum(g[:, s, None] * p[:, None, s] for s in range(4))
        w = shift(sum(np.conj(u[:, mu, None, b, :]) * h[:, :, b, None] for b in range(3)), DIMS, mu, -1)
        w[(t == 0) & (mu == 3)] *= -1
        ref += w
    ref = ref[orc.parity(DIMS) == 1]
    check(name, rms(out.download() - ref, ref))


def test_gauge_force(inputs):
    U = inputs[0]
    P = lqcd.momentum_field(DIMS).upload(np.zeros((V, 4, 8)))
    lqcd.gauge_force(P, lqcd.gauge_field(DIMS).upload(U), 6.0, 1.0)
    u, ref = U.astype(C), np.zeros((V, 4, 8), L)
    for mu in range(4):
        A = 0
        for nu in set(range(4)) - {mu}:
            ahead = shift(u[:, nu], DIMS, mu, 1)
            A = A + mm(mm(ahead, dag(shift(u[:, mu], DIMS, nu, 1))), dag(u[:, nu]))
            A = A + shift(mm(dag(mm(u[:, mu], ahead)), u[:, nu]), DIMS, nu, -1)
        w = mm(u[:, mu], A)
        for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
            ref[:, mu, a] = w[:, j, i].imag + w[:, i, j].imag
            ref[:, mu, a + 1] = w[:, i, j].real - w[:, j, i].real
        ref[:, mu, 2] = w[:, 0, 0].imag - w[:, 1, 1].imag
        ref[:, mu, 7] = (w[:, 0, 0].imag + w[:, 1, 1].imag - 2 * w[:, 2, 2].imag) / np.sqrt(L(3))
    check("gauge_force", rms(P.download() + ref, ref))


@pytest.mark.parametrize("c", [0.02, 0.1, 0.4, 0.7, 1.0, 4.0])
def test_link_update(inputs, c):
    U, _, P = inputs
    G = lqcd.gauge_field(DIMS).upload(U)
    lqcd.link_update(G, lqcd.momentum_field(DIMS).upload(P), c)
    n, p = 512, P[:512].astype(L) * (L(c) / 2)
    h = np.zeros((n, 4, 3, 3), C)
    for a, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        h[..., i, j], h[..., j, i] = p[..., a] - 1j * p[..., a + 1], p[..., a] + 1j * p[..., a + 1]
    d = p[..., 7] / np.sqrt(L(3))
    h[..., 0, 0], h[..., 1, 1], h[..., 2, 2] = p[..., 2] + d, -p[..., 2] + d, -2 * d
    halvings = 0
    while 3 * np.abs(h).max() > 0.25 * 2 ** halvings:
        halvings += 1
    x, eye = h * (C(1j) / 2 ** halvings), np.eye(3, dtype=C)
    e = eye + x / 16
    for k in range(15, 0, -1):  # Taylor series, remainder (1/4)^17 / 17!
        e = eye + mm(x, e) / k
    for _ in range(halvings):
        e = mm(e, e)
    ref = mm(e, U[:n].astype(C))
    check(c, rms(G.download()[:n] - ref, ref))


def test_reunitarize(inputs):
    U = inputs[0].copy()
    U[..., :2, :] = U[..., :2, :].real.astype(np.float16) + 1j * U[..., :2, :].imag.astype(np.float16)
    G = lqcd.gauge_field(DIMS).upload(U)
    lqcd.reunitarize(G)

    def norm(a):
        return np.sqrt((a.real ** 2 + a.imag ** 2).sum(-1, keepdims=True))

    r0, r1 = U[..., 0, :].astype(C), U[..., 1, :].astype(C)
    r0 = r0 / norm(r0)
    r1 = r1 - (np.conj(r0) * r1).sum(-1, keepdims=True) * r0
    r1 = r1 / norm(r1)
    out = G.download()
    check("row1", rms(out[..., 1, :] - r1))
    check("row2", rms(out[..., 2, :] - np.conj(np.cross(r0, r1))))


def test_plaquette():
    """over links of many 2^4 lattices, whose sums are short enough to show it"""
    dims, n, v = (2, 2, 2, 2), 2000, 16
    r = np.random.default_rng(7)
    got, U = [], []
    for _ in range(n):
        U.append(rand_su3(r, v * 4).reshape(v, 4, 3, 3))
        got.append(lqcd.plaquette(lqcd.gauge_field(dims).upload(U[-1])))
    u, s = np.array(U).astype(C), np.zeros(n, L)
    ahead = [np.roll(u.reshape(n, 2, 2, 2, 2, 4, 3, 3), -1, axis=4 - mu).reshape(u.shape) for mu in range(4)]
    for mu in range(4):
        for nu in range(mu + 1, 4):
            a, b = mm(u[:, :, mu], ahead[mu][:, :, nu]), mm(u[:, :, nu], ahead[nu][:, :, mu])
            s += (a.real * b.real + a.imag * b.imag).sum(axis=(1, 2, 3)) / 3
    check("plaquette", rms(np.array(got).astype(L) * 6 * v - s))
