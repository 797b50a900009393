"""Calls whose input lies in their output's memory (GPU).

The operator on axis-aligned cells reads cells that other blocks write the
result of, and so does the restriction by bricks.  Where a call takes vectors
that share memory, its result is the one of separate vectors, bit for bit.
"""
import pytest

import sipg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _vec(n, seed, dt=torch.float64):
    return torch.as_tensor(sipg_inputs.uniform(n, seed)).cuda().to(dt)


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("k", [1, 4])
def test_rows_shifted_by_one(k, dt):
    from paper_1910_01900_gb300 import Context
    ctx = Context((9, 10, 8), k)
    n, nv = ctx.num_dofs(), 5
    W = torch.stack([_vec(n, 10 + i, dt) for i in range(nv + 1)])
    want = torch.empty_like(W[:nv])
    ctx.apply_multi(W[:nv].clone(), want)
    torch.cuda.synchronize()
    ctx.apply_multi(W[:nv], W[1:])
    torch.cuda.synchronize()
    assert torch.equal(W[1:], want)


@pytest.mark.parametrize("deform", [0, 1])
def test_batch_round_robin(deform):
    """v[i] = A_i u[i] into the next problem's input, in a ring."""
    from paper_1910_01900_gb300 import Batch
    B = Batch([dict(m=(12, 9, 8), k=3, deform=deform) for _ in range(3)] + [dict(m=5, k=2, deform=deform)])
    x = [_vec(B.num_dofs(i), 20 + i) for i in range(4)]
    want = [torch.empty_like(t) for t in x]
    B.apply([t.clone() for t in x], want)
    torch.cuda.synchronize()
    last = torch.empty_like(x[3])
    B.apply(x, [x[1], x[2], x[0], last])
    torch.cuda.synchronize()
    assert torch.equal(x[1], want[0]) and torch.equal(x[2], want[1]) and torch.equal(x[0], want[2])
    assert torch.equal(last, want[3])


@pytest.mark.parametrize("deform", [0, 1])
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_timed_apply_in_place(deform, dt):
    from paper_1910_01900_gb300 import Context
    ctx = Context((12, 9, 8), 3, deform=deform, operator_only=True)
    u = _vec(ctx.num_dofs(), 7, dt)
    want, tmp = torch.empty_like(u), torch.empty_like(u)
    ctx.apply(u, tmp)
    ctx.apply(tmp, want)
    torch.cuda.synchronize()
    ctx.time_apply(u, u, repeats=2)
    torch.cuda.synchronize()
    assert torch.equal(u, want)


@pytest.mark.parametrize("k,deform,precision", [(4, 0, 0), (4, 0, 1), (5, 1, 1), (7, 0, 0), (3, 0, 1)])
def test_restriction_into_its_input(k, deform, precision):
    from paper_1910_01900_gb300 import Context
    ctx = Context((8, 6, 8), k, deform=deform, precision=precision, lambda_override=2.0)
    dt = torch.float32 if precision else torch.float64
    for level in range(1, ctx.num_levels):
        r = _vec(ctx.num_dofs(level), 30 + level, dt)
        nc = ctx.num_dofs(level - 1)
        want = torch.empty(nc, dtype=dt, device="cuda")
        ctx.restrict(level, r.clone(), want)
        torch.cuda.synchronize()
        ctx.restrict(level, r, r[:nc])
        torch.cuda.synchronize()
        assert torch.equal(r[:nc], want), level
