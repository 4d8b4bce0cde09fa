"""GPU: the iterate after k CG steps, for k on both sides of the pairs of steps in which x is updated and of
the 8 steps of a captured graph, against a textbook CG with the oracle's operator.

FP64: k steps of CG on a system of condition below 100 agree to 1e-12 for k <= 17; FP32 to 1e-5.
"""
import numpy as np
import pytest
import torch

import oracle
from lqhelp import Handle, dev, host, rel_err
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu

DIMS, M = (4, 4, 2, 4), 0.3


def steps(A, b, n):
    """The CG iterates x_0 .. x_n."""
    x, r = np.zeros_like(b), b.copy()
    p, rr, xs = r.copy(), np.vdot(r, r).real, [np.zeros_like(b)]
    for _ in range(n):
        if rr > 0:
            q = A(p)
            al = rr / np.vdot(p, q).real
            x, r = x + al * p, r - al * q
            new = np.vdot(r, r).real
            p, rr = r + (new / rr) * p, new
        xs.append(x.copy())
    return xs


@pytest.mark.parametrize("prec,tol", [(lqcd.LQ_F64, 1e-12), (lqcd.LQ_F32, 1e-5)])
def test_iterate_after_k_steps(prec, tol):
    U = inputs.gauge_field(DIMS, "smooth", seed=1800)
    prm = oracle.params(DIMS, mass=M)
    b = np.stack([inputs.gaussian_spinor(64, seed=2800), np.zeros((64, 4, 3), complex),
                  inputs.gaussian_spinor(64, seed=2801)])
    want = [steps(lambda v: oracle.apply_normal(oracle.OP_WILSON_EO, v, U, prm), f, 17) for f in b]
    with Handle(DIMS, U, mass=M) as H:
        for k in (1, 2, 3, 4, 7, 8, 9, 10, 16, 17):
            bd = dev(b, prec)
            x = torch.full_like(bd, 5.0)
            cp = lqcd.make_cg_params(lqcd.LQ_OP_WILSON_EO_NORMAL, lqcd.LQ_CG_PLAIN, prec, nrhs=3, tol=1e-30, maxiter=k)
            rc, st = lqcd.cg_solve(H.h, x, bd, cp, check=False)
            assert rc == -5 and [s.iters for s in st][0] == k and st[1].iters == 0
            got = host(x)
            assert not got[1].any()
            for j in (0, 2):
                assert rel_err(got[j], want[j][k]) < tol, (k, j)


def test_right_hand_sides_that_end_in_the_even_and_the_odd_step():
    """Right-hand sides that converge after different numbers of steps keep what they had then."""
    U = inputs.gauge_field(DIMS, "unit")
    prm = oracle.params(DIMS, mass=M)
    # plane waves: eigenvectors of the free normal operator; sums of j of them take at most j steps
    g = inputs.gaussian_spinor(1, seed=2802)[0]
    full = np.zeros((5, 128, 4, 3), complex)
    x0 = np.arange(128) % 4
    x1 = np.arange(128) // 4 % 4
    for j in range(1, 6):
        for n in range(j):
            full[j - 1] += np.exp(2j * np.pi * (n % 3 * x0 + n // 3 * x1) / 4)[:, None, None] * g * (1 + n)
    b = np.stack([inputs.to_half(f, DIMS, 0) for f in full])
    with Handle(DIMS, U, mass=M) as H:
        bd = dev(b)
        x = torch.empty_like(bd)
        cp = lqcd.make_cg_params(lqcd.LQ_OP_WILSON_EO_NORMAL, lqcd.LQ_CG_PLAIN, lqcd.LQ_F64, nrhs=5, tol=1e-10)
        rc, st = lqcd.cg_solve(H.h, x, bd, cp)
        got = host(x)
        assert rc == 0 and len({s.iters for s in st}) > 2
        for k in range(5):
            assert rel_err(oracle.apply_normal(oracle.OP_WILSON_EO, got[k], U, prm), b[k]) < 1e-10
