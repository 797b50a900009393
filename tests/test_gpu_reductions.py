"""Inner products of the flexible CG over vector lengths around the block counts.

The number of blocks follows the length (4096 entries per block, one block
without partials at the small end, a fixed maximum at the large one).  With
small whole numbers in b and a zero start vector the sum of squares is exact in
FP64 whatever the order, so the start residual's norm, the square root of that
sum, is known to the last bit, up to the rounding of the root itself.
"""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 64 entries; 4096, a block's share; 5832 and 8000, two blocks with a remainder;
# 125000, 31 blocks; 1.73 M, the maximum of 304 blocks
@pytest.mark.parametrize("m,k", [(2, 1), (4, 3), (3, 5), (5, 3), (10, 4), (24, 4)])
def test_start_residual_is_the_exact_sum(m, k):
    from paper_1910_01900_gb300 import Context
    ctx = Context(m=m, degree=k, deform=0, precision=0)
    n = ctx.num_dofs()
    g = torch.Generator().manual_seed(5)
    b = torch.randint(-9, 10, (n,), generator=g).double()
    want = math.sqrt(int((b.long() ** 2).sum()))
    bd, x = b.cuda(), torch.zeros(n, dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    info = ctx.solve(bd, x, rtol=1e-14, maxit=1, allow_notconv=True)
    assert abs(info.r0_norm - want) <= 2.3e-16 * want
    # the residual of the iterate by the plain operator: the update's own sum
    v = torch.empty_like(x)
    ctx.apply(x, v)
    torch.cuda.synchronize()
    r = float(torch.linalg.norm((bd - v).cpu()))
    assert abs(info.r_norm - r) <= 1e-11 * want
    ctx.close()
