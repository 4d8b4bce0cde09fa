"""GPU: the 5th-dimension kernels at slice counts around their batches of 6, against the oracle.

Tolerances of test_gpu_wilson.py: FP64 1e-12, FP32 2e-6 norm-wise; the Schur complement is two hops and
one 5th-dimension inverse of condition about 4: 1e-5 for FP32.
"""
import numpy as np
import pytest
import torch

import oracle
from lqhelp import Handle, dev, host, rel_err
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu

DIMS, V = (2, 4, 2, 4), 64


@pytest.mark.parametrize("Ls", [5, 6, 7, 12, 13])
@pytest.mark.parametrize("prec", [lqcd.LQ_F64, lqcd.LQ_F32])
@pytest.mark.parametrize("dag", [False, True])
def test_operators(Ls, prec, dag):
    U = inputs.gauge_field(DIMS, "random", seed=1700)
    psi = np.stack([inputs.gaussian_spinor(V, seed=2700 + s) for s in range(Ls)])
    half = np.stack([inputs.to_half(f, DIMS, 0) for f in psi])
    for mobius in (False, True):
        kw = dict(mobius=True, b5=1.5, c5=0.5) if mobius else {}
        with Handle(DIMS, U, Ls=Ls, M5=1.8, mf=0.1, **kw) as H:
            x = dev(psi, prec)
            y = torch.empty_like(x)
            lqcd.dwf_dslash_apply(H.h, y, x, prec, dag)
            want = (oracle.dwf_mobius_dslash(psi, U, DIMS, Ls, 1.8, 0.1, 1.5, 0.5, dagger=dag) if mobius
                    else oracle.dwf_dslash(psi, U, DIMS, Ls, 1.8, 0.1, dagger=dag))
            assert rel_err(host(y), want) < (1e-12 if prec == lqcd.LQ_F64 else 2e-6)
            x = dev(half, prec)
            y = torch.empty_like(x)
            lqcd.dwf_schur_apply(H.h, y, x, prec, dag)
            want = (oracle.dwf_mobius_schur(half, U, DIMS, Ls, 1.8, 0.1, 1.5, 0.5, dagger=dag) if mobius
                    else oracle.dwf_schur(half, U, DIMS, Ls, 1.8, 0.1, dagger=dag))
            assert rel_err(host(y), want) < (1e-12 if prec == lqcd.LQ_F64 else 1e-5)
