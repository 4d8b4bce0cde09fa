"""GPU: the FP64 SU(3) product real by real.

Bound: the a-priori one of FP64, u = 2^-53 times 6 (a sum of six products) times the sum of the six
products' absolute values, and for the subnormal range six units of 2^-1074.
"""
import numpy as np
import pytest
import torch

from lqhelp import ensure_built
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu


def check(A, B):
    ensure_built()
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    c = torch.empty_like(a)
    lqcd.lq_su3_mul(c, a, b, len(A), lqcd.LQ_F64)
    torch.cuda.synchronize()
    c = c.cpu().numpy()
    ar, ai, br, bi = (x.astype(np.longdouble) for x in (A.real, A.imag, B.real, B.imag))

    def dot(x, y):
        return sum(x[:, :, None, k] * y[:, None, k, :] for k in range(3))

    tol = 6.01 * np.longdouble(2.0) ** -53
    tiny = 6 * np.longdouble(2.0) ** -1074
    absr, absi = (np.abs(ar), np.abs(ai)), (np.abs(br), np.abs(bi))
    assert (np.abs(c.real - (dot(ar, br) - dot(ai, bi)))
            <= tol * (dot(absr[0], absi[0]) + dot(absr[1], absi[1])) + tiny).all()
    assert (np.abs(c.imag - (dot(ar, bi) + dot(ai, br)))
            <= tol * (dot(absr[0], absi[1]) + dot(absr[1], absi[0])) + tiny).all()


@pytest.mark.parametrize("eps", [1e-1, 1e-2, 1e-3, 1e-4, 1e-6, 1e-8, 1e-10, 1e-12, 1e-14, 1e-16, 1e-18, 1e-30])
def test_near_the_identity(eps):
    """exp(eps K), K antihermitian, as link updates have: real antisymmetric, imaginary symmetric, and both."""
    rng = np.random.default_rng(3800)
    r = rng.normal(size=(2, 129, 3, 3))
    for re, im in ((1, 0), (0, 1), (1, 1)):
        K = re * (r - r.transpose(0, 1, 3, 2)) + 1j * im * (r + r.transpose(0, 1, 3, 2))
        X = np.eye(3) + eps * K + eps * eps / 2 * (K @ K)
        X /= np.maximum(1, np.maximum(np.abs(X.real), np.abs(X.imag)).max((2, 3)))[..., None, None]
        check(X[0], X[1])
        check(X[0], inputs.random_su3(129, rng))
        check(inputs.random_su3(129, rng), X[0])


@pytest.mark.parametrize("n", [1, 31, 128, 129, 5001])
def test_random(n):
    rng = np.random.default_rng(3801)
    for make in (inputs.random_su3, inputs.smooth_su3):
        check(make(n, rng), make(n, rng))


@pytest.mark.parametrize("small", [1e-3, 1e-9, 1e-17, 1e-170, 5e-324])
def test_entries_of_different_size(small):
    """Entries of A and B scaled at random by 1 or `small`, zeros among them."""
    rng = np.random.default_rng(3802)
    A, B = inputs.random_su3(4001, rng), inputs.random_su3(4001, rng)
    for X in (A, B):
        v = X.view(np.float64)
        s = rng.integers(0, 5, v.shape)
        v[s == 0] *= small
        v[s == 1] = 0
    check(A, B)


def test_diagonal_matrices():
    n, rng = 257, np.random.default_rng(3803)
    D = np.zeros((n, 3, 3), complex)
    D[:, [0, 1, 2], [0, 1, 2]] = np.exp(1j * rng.uniform(0, 6.3, (n, 3)))
    one = np.tile(np.eye(3, dtype=complex), (n, 1, 1))
    for X in (one, D):
        check(X, D)
        check(X, inputs.random_su3(n, rng))
        check(inputs.random_su3(n, rng), X)
