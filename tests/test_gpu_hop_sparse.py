"""GPU: the FP64 hop on fields that are zero nearly everywhere (point and wall sources): the result, and that
zeros cost no more than other numbers.
"""
import numpy as np
import pytest
import torch

import oracle
from lqhelp import Handle, dev, host, native_buffer, rel_err
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dag", [False, True])
def test_zero_and_point_fields(dag):
    dims, V = (4, 6, 2, 4), 192
    U = inputs.gauge_field(dims, "random", seed=3600)
    fn = lqcd.dslash_dag_apply if dag else lqcd.dslash_apply
    with Handle(dims, U, mass=0.05) as H:
        for b in [np.zeros((V, 4, 3), complex), *inputs.point_sources(V, site=77)[[0, 4, 11]]]:
            x = dev(b)
            y = torch.empty_like(x)
            fn(H.h, y, x, lqcd.LQ_F64, lqcd.LQ_FULL)
            want = oracle.wilson_dslash(b, U, dims, 0.05, dagger=dag)
            assert not b.any() or rel_err(host(y), want) < 1e-15
            assert not host(y)[~want.any((1, 2))].any()


def test_subnormal_fields():
    """Neighbours whose high words are zero are not zero: unit links on small integers in units of 2^-1074."""
    dims, V = (4, 4, 2, 4), 128
    psi = np.random.default_rng(3).integers(-40, 41, (V, 4, 3, 2)) * 2.0
    psi[::3] = 0
    want = oracle.wilson_dslash(psi.view(np.complex128)[..., 0], inputs.gauge_field(dims, "unit"), dims, -4.0)
    with Handle(dims, inputs.gauge_field(dims, "unit"), mass=-4.0) as H:
        x = dev(np.ldexp(psi, -1074).view(np.complex128)[..., 0])
        y = torch.empty_like(x)
        lqcd.dslash_apply(H.h, y, x, lqcd.LQ_F64, lqcd.LQ_FULL)
        got = np.ascontiguousarray(host(y)).view(np.float64)
    assert np.array_equal(got, np.ldexp(np.ascontiguousarray(want).view(np.float64), -1074))


def microseconds(fn):
    best = 1e30
    for _ in range(5):
        fn()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(5):
            fn()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 200)
    return best


def test_zeros_cost_no_more():
    """A point source takes at most twice the time of a dense field (some sites around it take FP64 sums,
    a chain of 27 us or more whatever the lattice: 1.44 times here)."""
    dims = (16, 16, 32, 32)
    V = int(np.prod(dims))
    fmt = lqcd.LQ_NATIVE | lqcd.LQ_F64
    with Handle(dims, inputs.gauge_field(dims, "smooth", seed=3601), mass=0.05) as H:
        t = []
        for b in (inputs.gaussian_spinor(V, seed=3602), inputs.point_sources(V, site=5)[0]):
            x = native_buffer(H.h, lqcd.LQ_F64)
            lqcd.lq_convert(H.h, x, fmt, dev(b), lqcd.LQ_F64)
            y = torch.empty_like(x)
            t.append(microseconds(lambda: lqcd.dslash_apply(H.h, y, x, fmt, lqcd.LQ_FULL)))
        assert t[1] < 2 * t[0], t
