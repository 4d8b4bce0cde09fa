"""GPU: the FP64 hop with links that are not SU(3): of a smaller scale, in part or as a whole, and zero.

The hop alone (LQ_EVEN, or m = -4), compared colour by colour.  Tolerance 1e-15 of the colour's norm, as
in test_gpu_hop_fixed.py: FP64 products and sums, whatever the links' scale.
"""
import numpy as np
import pytest
import torch

import oracle
from lqhelp import Handle, dev, host, rel_err
from paper_2001_07557_gb300 import inputs, lqcd


pytestmark = pytest.mark.gpu

DIMS, V = (4, 6, 2, 4), 192


def check(U):
    psi = inputs.gaussian_spinor(V, seed=3500)
    odd = inputs.to_half(psi, DIMS, 1)
    with Handle(DIMS, U, mass=-4.0) as H:
        for dag in (False, True):
            fn = lqcd.dslash_dag_apply if dag else lqcd.dslash_apply
            for x, parity, want in (
                    (odd, lqcd.LQ_EVEN, -0.5 * oracle.wilson_hop_eo(odd, U, DIMS, 0, dagger=dag)),
                    (psi, lqcd.LQ_FULL, oracle.wilson_dslash(psi, U, DIMS, -4.0, dagger=dag))):
                xd = dev(x)
                y = torch.empty_like(xd)
                fn(H.h, y, xd, lqcd.LQ_F64, parity)
                got = host(y)
                for c in range(3):
                    if not want[..., c].any():
                        assert not got[..., c].any()
                    else:
                        assert rel_err(got[..., c], want[..., c]) < 1e-15, (parity, dag, c)


@pytest.mark.parametrize("scale", [0.2, 1e-3, 1e-6, 1e-9, 1e-12, 2.0 ** -60, 1e-100])
def test_links_of_a_smaller_scale(scale):
    check(scale * inputs.gauge_field(DIMS, "random", seed=3501))


@pytest.mark.parametrize("scale", [1e-4, 1e-9, 2.0 ** -60])
def test_one_small_colour(scale):
    """diag(1, 1, s) and its like leave every link with entries of both scales."""
    U = inputs.gauge_field(DIMS, "unit")
    U[:, :, 2, 2] = scale
    check(U)


def test_zero_links():
    """Open boundary in time: the links across it are zero."""
    U = inputs.gauge_field(DIMS, "random", seed=3502)
    U.reshape(4, 2, 6, 4, 4, 3, 3)[3, :, :, :, 3] = 0
    check(U)
    check(np.zeros_like(U))
