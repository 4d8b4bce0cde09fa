"""GPU: the FP64 hop in 64-bit fixed point (hop_fixed.cuh) against the FP64 oracle, and the rule that
keeps the FP64 kernel for links it cannot take.

Tolerance: the fixed-point sums carry 56 or more bits below the largest neighbour component and are
rounded to FP64 once (2^-53); the oracle and the FP64 kernel round about 60 partial sums, none above
39 times that component.  1e-15 norm-wise holds both.
"""
import numpy as np
import pytest
import torch

import oracle
from lqhelp import Handle, dev, host, rel_err
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu

BC = (-1, 1, 1, -1)
F64 = lqcd.LQ_F64


def apply(H, x, parity, dag, nrhs=1):
    xd = dev(x)
    y = torch.empty_like(xd)
    (lqcd.dslash_dag_apply if dag else lqcd.dslash_apply)(H.h, y, xd, F64, parity, nrhs)
    return host(y)


# 8, 96, 120 and 192 sites of a parity: below, and no multiple of, a warp's 16 and a block's 128
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 4, 2), (10, 2, 6, 2), (4, 6, 2, 8)])
@pytest.mark.parametrize("dag", [False, True])
@pytest.mark.parametrize("unfit", [False, True])
def test_every_form_against_the_oracle(dims, dag, unfit):
    V, m, n = int(np.prod(dims)), 0.05, 3
    U = inputs.gauge_field(dims, "random", seed=1500)
    if unfit:  # one entry above 1: the handle keeps the FP64 kernel
        U[V // 2, 1, 0, 0] = 1.5
    psi = np.stack([inputs.gaussian_spinor(V, seed=2500 + k) for k in range(n)])
    half = [np.stack([inputs.to_half(f, dims, p) for f in psi]) for p in (0, 1)]
    with Handle(dims, U, mass=m, bc=BC) as H:
        want = np.stack([oracle.wilson_dslash(f, U, dims, m, bc=BC, dagger=dag) for f in psi])
        assert rel_err(apply(H, psi, lqcd.LQ_FULL, dag, n), want) < 1e-15
        for p in (0, 1):
            want = np.stack([-0.5 * oracle.wilson_hop_eo(f, U, dims, p, bc=BC, dagger=dag) for f in half[1 - p]])
            assert rel_err(apply(H, half[1 - p], p, dag, n), want) < 1e-15
        want = np.stack([oracle.wilson_schur(f, U, dims, m, bc=BC, dagger=dag) for f in half[0]])
        assert rel_err(apply(H, half[0], lqcd.LQ_SCHUR_EVEN, dag, n), want) < 2e-15  # two hops


@pytest.mark.parametrize("Ls", [1, 5])
@pytest.mark.parametrize("dag", [False, True])
def test_domain_wall(Ls, dag):
    dims = (6, 4, 4, 2)
    U = inputs.gauge_field(dims, "random", seed=1501)
    psi = np.stack([inputs.gaussian_spinor(192, seed=2510 + k) for k in range(Ls)])
    with Handle(dims, U, bc=BC, Ls=Ls, M5=1.8, mf=0.1) as H:
        x = dev(psi)
        y = torch.empty_like(x)
        lqcd.dwf_dslash_apply(H.h, y, x, F64, dag)
        assert rel_err(host(y), oracle.dwf_dslash(psi, U, dims, Ls, 1.8, 0.1, bc=BC, dagger=dag)) < 1e-15


# block exponents inside the fixed-point range, at its ends, and outside on both sides (subnormal results
# at 2^-1060 keep 14 bits)
@pytest.mark.parametrize("k,tol", [(0, 1e-15), (-880, 1e-15), (-900, 1e-15), (960, 1e-15), (985, 1e-15),
                                   (1010, 1e-15), (-1060, 1e-4)])
def test_scaled_fields(k, tol):
    dims = (4, 4, 2, 4)
    U = inputs.gauge_field(dims, "random", seed=1502)
    psi = inputs.gaussian_spinor(128, seed=2520)
    want = oracle.wilson_dslash(psi, U, dims, 0.05)
    with Handle(dims, U, mass=0.05) as H:
        got = apply(H, np.ldexp(psi.view(np.float64), k).view(np.complex128), lqcd.LQ_FULL, False)
    assert rel_err(np.ldexp(got.view(np.float64), -k).view(np.complex128), want) < tol


def test_mixed_magnitudes():
    """Sites whose scales differ by up to 2^40: each output is accurate to its largest neighbour."""
    dims = (4, 4, 4, 4)
    U = inputs.gauge_field(dims, "random", seed=1503)
    e = np.random.default_rng(5).integers(-20, 21, 256)
    psi = inputs.gaussian_spinor(256, seed=2530) * np.ldexp(1.0, e)[:, None, None]
    hop = oracle.wilson_dslash(psi, U, dims, -4.0)
    with Handle(dims, U, mass=-4.0) as H:
        got = apply(H, psi, lqcd.LQ_FULL, False)
    x = np.stack([np.abs(psi).max((1, 2)).reshape(4, 4, 4, 4)])[0]
    big = np.max([np.roll(x, s, a) for a in range(4) for s in (1, -1)], axis=0).reshape(-1)
    assert np.max(np.abs(got - hop).max((1, 2)) / big) < 4e-15


def test_exact_on_dyadic_numbers():
    """Unit links, m = 0 and a point source: every sum is exact, zeros among them."""
    dims = (4, 4, 4, 4)
    U = inputs.gauge_field(dims, "unit")
    with Handle(dims, U, mass=0.0) as H:
        for b in inputs.point_sources(256, site=37)[[0, 5, 11]]:
            for dag in (False, True):
                assert np.array_equal(apply(H, b, lqcd.LQ_FULL, dag), oracle.wilson_dslash(b, U, dims, 0.0, dagger=dag))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_input_stays_with_its_neighbours(bad):
    dims = (4, 4, 4, 4)
    U = inputs.gauge_field(dims, "random", seed=1504)
    psi = inputs.gaussian_spinor(256, seed=2540)
    clean = psi.copy()
    clean[100] = 0
    psi[100, 2, 1] = bad
    want = oracle.wilson_dslash(clean, U, dims, -4.0)  # the hop alone: site 100 reaches its neighbours only
    at = np.zeros((4, 4, 4, 4), bool)
    at.reshape(-1)[100] = True
    touched = np.any([np.roll(at, s, a) for a in range(4) for s in (1, -1)], axis=0).reshape(-1)
    with Handle(dims, U, mass=-4.0) as H:
        got = apply(H, psi, lqcd.LQ_FULL, False)
    far = ~touched
    far[100] = False  # 0 times the bad value
    assert not np.isfinite(got[touched]).all(axis=(1, 2)).any()
    assert rel_err(got[far], want[far]) < 1e-15
