"""GPU: a solve that has no room for its second search direction takes one, with the same iterates."""
import pytest
import torch

from lqhelp import Handle, dev
from paper_2001_07557_gb300 import inputs, lqcd

pytestmark = pytest.mark.gpu

DIMS, V = (16, 16, 16, 32), 16 ** 3 * 32


def solve(H, b, mode):
    x = torch.zeros_like(b)
    cp = lqcd.make_cg_params(lqcd.LQ_OP_WILSON_EO_NORMAL, mode, lqcd.LQ_F64, nrhs=4, tol=1e-10, inner=lqcd.LQ_F32)
    free = torch.cuda.mem_get_info()[0]
    rc, st = lqcd.cg_solve(H.h, x, b, cp)
    assert rc == 0
    return x, [s.iters for s in st], free - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("mode,vector", [(lqcd.LQ_CG_PLAIN, 192), (lqcd.LQ_CG_BATCHED, 96)])
def test_solve_without_room_for_two_search_directions(mode, vector):
    U = inputs.gauge_field(DIMS, "smooth", seed=1900)
    b = dev(inputs.gaussian_spinor(V // 2, seed=2900, nrhs=4))
    size = 4 * (V // 2) * vector  # of the search directions
    with Handle(DIMS, U, mass=0.1) as H:  # the first loads the kernels
        solve(H, b, mode)
    with Handle(DIMS, U, mass=0.1) as H:
        x, iters, used = solve(H, b, mode)
        torch.cuda.empty_cache()
    assert used > size
    with Handle(DIMS, U, mass=0.1) as H:
        room = [torch.empty_like(x) for _ in range(2)]  # for the solutions that solve() allocates
        del room
        filler = torch.empty(torch.cuda.mem_get_info()[0] - used + size // 2, dtype=torch.uint8, device="cuda")
        y, again, _ = solve(H, b, mode)  # all but half of a vector fits
        z, third, _ = solve(H, b, mode)
        del filler
    torch.cuda.empty_cache()
    assert again == iters == third and torch.equal(x, y) and torch.equal(x, z)
