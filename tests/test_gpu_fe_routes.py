"""The FE operator on axis-aligned cells where its route changes (GPU).

In FP64 some sizes of a degree take the cell and node passes and the others the
one pass over bricks.  Meshes on both sides of every line against the general
path (the same mesh as a deformed one of amplitude 0; FP64 <= 1e-12, the bound of the
operator parity tests), and a batch whose problems take both routes against
each problem's own cycle, bit for bit.
"""
import pytest

import sipg_inputs
from parity_check import close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (0, 1, 1, 0, 0, 0)

CASES = [((9, 11, 10), 2), ((10, 10, 10), 2), ((17, 17, 17), 2), ((17, 17, 18), 2), ((7, 6, 7), 3), ((7, 7, 7), 3),
         ((12, 12, 13), 3), ((13, 13, 12), 3), ((5, 6, 6), 4), ((7, 5, 6), 4), ((22, 23, 23), 4), ((23, 23, 23), 4),
         ((1, 1, 1), 5), ((5, 3, 7), 5), ((4, 3, 2), 6), ((2, 5, 3), 7), ((3, 2, 3), 8)]


@pytest.mark.parametrize("m,k", CASES)
def test_fe_operator_on_both_sides_of_the_line(m, k):
    from paper_1910_01900_gb300 import Context
    box, general = (Context(m, k, bc=BC, fe_assemble=0, lambda_override=2.0, **kw)
                    for kw in (dict(), dict(deform=1, amp=0.0)))
    level = box.num_levels - 2
    u = torch.as_tensor(sipg_inputs.uniform(box.num_dofs(level), 50 + k)).cuda()
    v, ref = torch.full_like(u, float("nan")), torch.empty_like(u)
    box.level_apply(level, u, v)
    general.level_apply(level, u, ref)
    torch.cuda.synchronize()
    assert close(v.cpu().numpy(), ref.cpu().numpy()) <= 1e-12
    for cb in (1, 3, 7):   # the width changes the launch, not the sums
        box.set_tile_shape(0, 2, cb, level=level)
        w = torch.full_like(u, float("nan"))
        box.level_apply(level, u, w)
        torch.cuda.synchronize()
        assert torch.equal(v, w), cb


def test_batch_with_both_routes_equals_each_problems_cycle():
    from paper_1910_01900_gb300 import Batch
    probs = [dict(m=m, k=k) for m, k in ((10, 2), (4, 2), (7, 3), ((4, 3, 5), 3), (6, 4), (4, 4), (4, 5), (3, 6))]
    s = torch.cuda.Stream()
    B = Batch(probs, stream=s)
    rs = [torch.as_tensor(sipg_inputs.uniform(B.num_dofs(i), 90 + i)).cuda() for i in range(len(probs))]
    zs = [torch.full_like(r, float("nan")) for r in rs]
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        B.vcycle(rs, zs)
    torch.cuda.synchronize()
    for i, r in enumerate(rs):
        z = torch.empty_like(r)
        B.contexts[i].vcycle(r, z)
        torch.cuda.synchronize()
        assert torch.equal(zs[i], z), probs[i]


def test_widths_of_an_fe_level_are_the_cells_of_its_bricks():
    """The default width is the cells of the brick that runs (4 x 4 x 2 of degree 4 here), it
    can be set again although no other width above the limit can, and the full brick with a
    remainder in every direction gives the general path's result in FP32 too."""
    from paper_1910_01900_gb300 import Context
    from paper_1910_01900_gb300.csrc_info import max_cells_per_block
    from paper_1910_01900_gb300.native import SipgError
    m, k = (21, 22, 11), 4
    box, general = (Context(m, k, bc=BC, fe_assemble=0, lambda_override=2.0, **kw)
                    for kw in (dict(), dict(deform=1, amp=0.0)))
    level = box.num_levels - 2
    assert box.tile_shape(1, 2, level) == 32 > max_cells_per_block(k + 1, 4)
    u = torch.as_tensor(sipg_inputs.uniform(box.num_dofs(level), 5)).cuda()
    ref = torch.empty_like(u)
    general.level_apply(level, u, ref)
    first = None
    for cb in (0, 10, 1, 32):
        box.set_tile_shape(1, 2, cb, level=level)
        assert box.tile_shape(1, 2, level) == (cb or 32)
        v = torch.full_like(u, float("nan"), dtype=torch.float32)
        box.level_apply(level, u.float(), v)
        torch.cuda.synchronize()
        if first is None:
            first = v
            assert close(v.cpu().numpy().astype("float64"), ref.cpu().numpy()) <= 1e-5
        assert torch.equal(v, first), cb
    with pytest.raises(SipgError):
        box.set_tile_shape(1, 2, 31, level=level)


@pytest.mark.parametrize("k", [2, 4, 6])
def test_autotuned_fe_levels_give_the_same_results(k):
    from paper_1910_01900_gb300 import Context
    m = (9, 10, 12)
    plain, tuned = (Context(m, k, bc=BC, fe_assemble=0, lambda_override=2.0, autotune=a) for a in (False, True))
    for level in range(1, plain.num_levels - 1):
        for dt, prec in ((torch.float64, 0), (torch.float32, 1)):
            u = torch.as_tensor(sipg_inputs.uniform(plain.num_dofs(level), 40 + level)).cuda().to(dt)
            v, w, x = (torch.full_like(u, float("nan")) for _ in range(3))
            plain.level_apply(level, u, v)
            tuned.level_apply(level, u, w)
            width = tuned.tile_shape(prec, 2, level)
            tuned.set_tile_shape(prec, 2, width, level=level)   # a tuned width can be set again
            assert tuned.tile_shape(prec, 2, level) == width
            tuned.level_apply(level, u, x)
            torch.cuda.synchronize()
            assert torch.equal(v, w) and torch.equal(v, x), (level, prec)
