"""The p- and c-transfers on both sides of the sizes where their kernel changes (GPU).

The general kernels and the ones by bricks (or lines) of cells compute the same
sums, so on meshes just below and just above each line both are compared with
the 1D interpolation matrices applied axis by axis in 64 bits (FP64 <= 1e-12,
FP32 <= 1e-5, the bounds of the transfer parity tests).
"""
import numpy as np
import pytest

import sipg_inputs
from oracle.basis import gauss_lobatto, lagrange_values
from parity_check import close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
BC = (0, 1, 1, 0, 0, 0)


def _global_1d(m, pf, pc):
    local = lagrange_values(gauss_lobatto(pc + 1), gauss_lobatto(pf + 1))
    P = np.zeros((m * pf + 1, m * pc + 1))
    for c in range(m):
        P[c * pf:(c + 1) * pf + 1, c * pc:(c + 1) * pc + 1] = local
    return P


def _free(m, p):
    """1 on the free nodes of the grid [z][y][x], 0 on the Dirichlet ones."""
    f = np.ones([m[a] * p + 1 for a in (2, 1, 0)])
    for d in range(3):
        for s in range(2):
            if BC[2 * d + s] == 0:
                np.moveaxis(f, 2 - d, 0)[-1 if s else 0] = 0
    return f


def _along(U, mats):   # mats of x, y, z
    for ax, M in zip((2, 1, 0), mats):
        U = np.moveaxis(np.tensordot(M, U, axes=(1, ax)), 0, ax)
    return U


CASES = [(3, 0, (20, 20, 20)), (3, 0, (19, 20, 20)), (3, 1, (31, 31, 31)), (3, 1, (30, 30, 32)),
         (4, 0, (8, 9, 9)), (4, 0, (8, 8, 9)), (4, 1, (14, 15, 15)), (4, 1, (14, 14, 15)),
         (5, 1, (8, 8, 8)), (5, 1, (7, 8, 9)), (6, 0, (20, 20, 20)), (6, 0, (19, 20, 20)),
         (7, 1, (8, 8, 8)), (7, 1, (7, 8, 9)), (7, 0, (5, 3, 4)), (8, 0, (5, 3, 4))]


@pytest.mark.parametrize("k,precision,m", CASES)
def test_p_transfers_on_both_sides_of_the_line(k, precision, m):
    from paper_1910_01900_gb300 import Context
    ctx = Context(m, k, bc=BC, precision=precision, lambda_override=2.0)
    fine, pc, tol = ctx.num_levels - 2, k // 2, 1e-5 if precision else 1e-12
    assert ctx.level_info(fine - 1)[:2] == (1, pc)
    dt = torch.float32 if precision else torch.float64
    P = [_global_1d(m[a], k, pc) for a in range(3)]
    ff, fc = _free(m, k), _free(m, pc)
    r, x = (sipg_inputs.uniform(ff.size, 60 + k + i).reshape(ff.shape) for i in range(2))
    xc = sipg_inputs.uniform(fc.size, 80 + k).reshape(fc.shape) * fc
    rc = torch.full((fc.size,), float("nan"), dtype=dt, device="cuda")
    xg = torch.as_tensor(x.ravel()).cuda().to(dt)
    ctx.restrict(fine, torch.as_tensor(r.ravel()).cuda().to(dt), rc)
    ctx.prolongate_add(fine, torch.as_tensor(xc.ravel()).cuda().to(dt), xg)
    torch.cuda.synchronize()
    assert close(rc.cpu().numpy().astype(np.float64), (fc * _along(r * ff, [M.T for M in P])).ravel()) <= tol
    assert close(xg.cpu().numpy().astype(np.float64), (x + ff * _along(xc, P)).ravel()) <= tol


@pytest.mark.parametrize("k,m", [(5, (6, 8, 9)), (5, (6, 8, 10)), (8, (5, 5, 5)), (8, (5, 5, 6)), (4, (2, 3, 1))])
@pytest.mark.parametrize("precision", [0, 1])
def test_c_prolongation_on_both_sides_of_the_line(k, precision, m):
    from paper_1910_01900_gb300 import Context
    ctx = Context(m, k, bc=BC, precision=precision, lambda_override=2.0)
    L = ctx.num_levels - 1
    dt = torch.float32 if precision else torch.float64
    xc = torch.as_tensor(sipg_inputs.uniform(ctx.num_dofs(L - 1), 5)).cuda().to(dt)
    x = torch.as_tensor(sipg_inputs.uniform(ctx.num_dofs(L), 6)).cuda().to(dt)
    free = torch.as_tensor(_free(m, k)).cuda().to(dt)
    U = xc.view(free.shape) * free
    cells = torch.stack([U[z * k:z * k + k + 1, y * k:y * k + k + 1, q * k:q * k + k + 1]
                         for z in range(m[2]) for y in range(m[1]) for q in range(m[0])])
    want = x + cells.reshape(-1)
    torch.cuda.synchronize()
    ctx.prolongate_add(L, xc, x)
    torch.cuda.synchronize()
    assert torch.equal(x, want)
