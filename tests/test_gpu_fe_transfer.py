"""The p-transfers by bricks of cells against the oracle (GPU).

Every pair of the default sequence p -> floor(p/2) that has a brick kernel, on
meshes whose sides leave odd bricks, with mixed boundary conditions: the
prolongation and the restriction against the oracle's assembled projection
(FP64 <= 1e-12, FP32 <= 1e-5), with vectors that are not zero on the
constrained nodes.
"""
import numpy as np
import pytest

import sipg_inputs
from oracle.fe import FESpace
from oracle.mesh import Mesh
from oracle.transfer import fe_transfer
from parity_check import close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [((6, 2, 5), 3, (0, 0, 1, 0, 0, 1)), ((5, 9, 3), 4, (0, 1, 0, 0, 1, 0)), ((9, 3, 1), 5, (1, 0, 0, 1, 0, 0)),
         ((4, 3, 5), 6, (0, 0, 0, 0, 0, 0)), ((3, 5, 2), 7, (0, 1, 1, 0, 0, 1)), ((1, 3, 5), 8, (0, 0, 1, 0, 0, 0))]


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
@pytest.mark.parametrize("m,k,bc", CASES)
def test_p_transfers_match_the_projection(m, k, bc, precision, tol):
    from paper_1910_01900_gb300 import Context
    ctx = Context(m, k, bc=bc, precision=precision, lambda_override=2.0)
    fine = ctx.num_levels - 2
    mesh = Mesh(m, bc=bc)
    P = fe_transfer(FESpace(mesh, k), FESpace(mesh, k // 2))
    dt = torch.float32 if precision else torch.float64
    r = sipg_inputs.uniform(ctx.num_dofs(fine), 60 + k)
    rc = torch.full((ctx.num_dofs(fine - 1),), float("nan"), dtype=dt, device="cuda")
    ctx.restrict(fine, torch.as_tensor(r).cuda().to(dt), rc)
    assert close(rc.cpu().numpy().astype(np.float64), P.T @ r) <= tol
    xc = sipg_inputs.uniform(ctx.num_dofs(fine - 1), 70 + k)
    x = sipg_inputs.uniform(ctx.num_dofs(fine), 80 + k)
    # the oracle's P ignores coarse values on constrained nodes, which a cycle keeps at zero
    xc[FESpace(mesh, k // 2).constrained] = 0.0
    xg = torch.as_tensor(x).cuda().to(dt)
    ctx.prolongate_add(fine, torch.as_tensor(xc).cuda().to(dt), xg)
    assert close(xg.cpu().numpy().astype(np.float64), x + P @ xc) <= tol
