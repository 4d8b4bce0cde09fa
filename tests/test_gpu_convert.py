"""GPU: native fields written back to site-major, at sizes around a warp's 32 and a block's 128 sites.

Values are such that every format holds them exactly (small integers over a site maximum that is a power
of two), so conversions must return them bit for bit.
"""
import numpy as np
import pytest
import torch

from lqhelp import Handle, native_buffer
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 2, 2), (2, 2, 2, 8), (10, 2, 6, 2), (2, 2, 2, 34), (2, 6, 2, 44)])
@pytest.mark.parametrize("prec", [lqcd.LQ_F64, lqcd.LQ_F32, lqcd.LQ_F16, lqcd.LQ_BF16])
@pytest.mark.parametrize("sm", [lqcd.LQ_F64, lqcd.LQ_F32])
@pytest.mark.parametrize("host_memory", [False, True])
def test_round_trip(dims, prec, sm, host_memory):
    V, n = int(np.prod(dims)), 3
    rng = np.random.default_rng(9)
    v = rng.integers(-63, 64, (n, V, 12, 2)).astype(np.float64)
    v[:, :, 5, 1] = 64
    v *= np.ldexp(1.0, rng.integers(-5, 6, (n, V)))[:, :, None, None]
    dt = torch.float64 if sm == lqcd.LQ_F64 else torch.float32
    with Handle(dims, inputs.gauge_field(dims, "unit")) as H:
        for subset in (lqcd.LQ_FULL, lqcd.LQ_EVEN, lqcd.LQ_ODD):
            sites = V if subset == lqcd.LQ_FULL else V // 2
            x = torch.from_numpy(np.ascontiguousarray(v[:, :sites])).to(dt).cuda()
            nat = native_buffer(H.h, prec, subset, n)
            y = torch.full_like(x, -1.0, device="cpu" if host_memory else "cuda")
            if host_memory:
                y = y.pin_memory()
            lqcd.lq_convert(H.h, nat, lqcd.LQ_NATIVE | prec, x, sm, subset, n)
            lqcd.lq_convert(H.h, y, sm, nat, lqcd.LQ_NATIVE | prec, subset, n)
            torch.cuda.synchronize()
            assert torch.equal(y.cpu(), x.cpu())
