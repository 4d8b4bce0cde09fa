"""GPU: launches of several right-hand sides whose blocks share the links (hop_shared.cuh), against
launches of one right-hand side each, bit for bit: the arithmetic is the same in the same order.

The counts lie on both sides of every line of the dispatch (one-right-hand-side kernel, three groups,
four groups) and leave whole and partial last rounds; the lattices have whole and ragged 32-site tiles.
"""
import numpy as np
import pytest
import torch

from lqhelp import Handle, dev, native_buffer
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (2, 6, 2, 6)])
@pytest.mark.parametrize("prec,r12", [(lqcd.LQ_F32, False), (lqcd.LQ_F32, True), (lqcd.LQ_F16, True),
                                      (lqcd.LQ_BF16, True)])
@pytest.mark.parametrize("dag", [False, True])
def test_equal_to_single_launches(dims, prec, r12, dag):
    V = int(np.prod(dims))
    fmt = lqcd.LQ_NATIVE | prec
    U = inputs.gauge_field(dims, "random", seed=1600)
    fn = lqcd.dslash_dag_apply if dag else lqcd.dslash_apply
    with Handle(dims, U, mass=0.05, bc=(-1, 1, 1, -1), compress12=r12) as H:
        for parity, subset, sites in ((lqcd.LQ_FULL, lqcd.LQ_FULL, V), (lqcd.LQ_ODD, lqcd.LQ_EVEN, V // 2),
                                      (lqcd.LQ_SCHUR_EVEN, lqcd.LQ_EVEN, V // 2)):
            x = dev(inputs.gaussian_spinor(sites, seed=2600, nrhs=13))
            xn = native_buffer(H.h, prec, subset, 13)
            lqcd.lq_convert(H.h, xn, fmt, x, lqcd.LQ_F64, subset, 13)
            one = native_buffer(H.h, prec, subset, 13).view(13, -1)
            for k in range(13):
                fn(H.h, one[k], xn.view(13, -1)[k], fmt, parity)
            for n in (2, 3, 4, 5, 6, 7, 9, 12, 13):
                y = native_buffer(H.h, prec, subset, n)
                fn(H.h, y, xn, fmt, parity, n)
                torch.cuda.synchronize()
                assert torch.equal(y.view(n, -1), one[:n]), (parity, n)
