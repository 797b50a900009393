"""FP32 rounding of the one-pass operator on axis-aligned cells (GPU).

The yardstick is the same operator evaluated at the Gauss points in FP32
(interpolation, metric, transposed interpolation, stored face traces), whose
relative error in the 2-norm against 64 bits for uniform random vectors is
measured per degree on meshes of about 1e6 points: the one-pass form must not
round more (2% for the spread between seeds and meshes).
"""
import pytest

import sipg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GAUSS_POINT_FORM = {1: 9.66e-8, 2: 1.541e-7, 3: 1.847e-7, 4: 1.927e-7, 5: 2.52e-7, 6: 2.167e-7, 7: 2.564e-7,
                    8: 2.436e-7}
SIDE = {1: 50, 2: 33, 3: 25, 4: 20, 5: 17, 6: 14, 7: 12, 8: 11}


@pytest.mark.parametrize("k", sorted(SIDE))
def test_one_pass_rounds_no_more_than_the_gauss_point_form(k):
    from paper_1910_01900_gb300 import Context
    ctx = Context(SIDE[k], k, operator_only=True)
    u = torch.as_tensor(sipg_inputs.uniform(ctx.num_dofs(), 70 + k)).cuda().float()
    v, ref = torch.empty_like(u), torch.empty(len(u), dtype=torch.float64, device=u.device)
    ctx.apply(u, v)
    ctx.apply(u.double(), ref)
    torch.cuda.synchronize()
    err = ((v.double() - ref).norm() / ref.norm()).item()
    assert err <= 1.02 * GAUSS_POINT_FORM[k], err
