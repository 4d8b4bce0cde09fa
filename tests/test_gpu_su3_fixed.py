"""GPU: the FP64 SU(3) product's fixed-point path against the FP64 unit's, matrix by matrix.

An entry of a fixed-point product is a sum exact to 2^-57 rounded once (2^-54 at most, as entries are
at most 1): 2e-16 with the reference's own rounding (2^-53 for sums of six).  Other matrices keep
the FP64 unit: 1e-14 of the largest entry, the tolerance of test_gpu_su3.py.
"""
import numpy as np
import pytest
import torch

from lqhelp import ensure_built
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu


def product(A, B):
    ensure_built()
    a, b = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    c = torch.empty_like(a)
    lqcd.lq_su3_mul(c, a, b, len(A), lqcd.LQ_F64)
    torch.cuda.synchronize()
    return c.cpu().numpy()


@pytest.mark.parametrize("n", [1, 31, 128, 129, 40001])
@pytest.mark.parametrize("kind", ["random", "smooth", "unit"])
def test_su3_matrices(n, kind):
    rng = np.random.default_rng(7)
    if kind == "unit":
        A, B = np.tile(np.eye(3, dtype=complex), (n, 1, 1)), inputs.random_su3(n, rng)
        assert np.array_equal(product(A, A), A)
    else:
        make = inputs.random_su3 if kind == "random" else inputs.smooth_su3
        A, B = make(n, rng), make(n, rng)
    assert np.max(np.abs(product(A, B) - np.matmul(A, B))) < 4e-16


def test_neighbouring_matrices_of_other_scales():
    """Within one warp: SU(3) pairs beside pairs too large, too small, with a zero row, and not finite."""
    n = 256
    rng = np.random.default_rng(8)
    A, B = inputs.random_su3(n, rng), inputs.random_su3(n, rng)
    A[3::16] *= 1e3
    B[5::16] *= 1e-200
    A[7::16, 1] = 0
    B[9::16, 0, 0] = 1.5
    A[11::16] *= 1e300
    with np.errstate(all="ignore"):
        want = np.matmul(A, B)
    got = product(A, B)
    scale = np.abs(want).max((1, 2))
    assert np.max(np.abs(got - want).max((1, 2)) / scale) < 1e-14
    for bad in (np.nan, np.inf):
        A[13, 2, 1] = bad
        got2 = product(A, B)
        assert not np.isfinite(got2[13, 2]).any() and np.array_equal(np.delete(got2, 13, 0), np.delete(got, 13, 0))
        assert np.array_equal(got2[13, :2], got[13, :2]) or np.allclose(got2[13, :2], got[13, :2], rtol=0, atol=4e-16)
