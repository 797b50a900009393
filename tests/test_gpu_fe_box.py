"""The one-pass FE operator on axis-aligned cells against the oracle (GPU).

A thread block computes the nodes of a brick of cells with one layer of cells
below it, so the sizes that matter are single cells, bricks that do not divide
the mesh and the mesh's last plane; each result is compared element by element
with the FP64 oracle (FP64 <= 1e-12, FP32 <= 1e-5, the bounds of the operator
parity tests) and bit for bit between bricks.
"""
import numpy as np
import pytest

import sipg_inputs
from oracle.fe import FESpace
from oracle.mesh import Mesh
from parity_check import close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # cells, degree, boundary codes (0 Dirichlet, 1 Neumann)
    ((1, 1, 1), 2, (0, 1, 0, 1, 0, 1)),
    ((1, 3, 2), 8, (0, 1, 1, 0, 0, 0)),
    ((9, 4, 5), 1, (0, 1, 0, 0, 1, 0)),
    ((7, 9, 3), 2, (1, 0, 0, 1, 0, 0)),
    ((6, 2, 5), 3, (0, 0, 1, 0, 0, 1)),
    ((5, 3, 4), 4, (0, 0, 0, 0, 0, 0)),
    ((4, 1, 5), 5, (0, 1, 0, 0, 1, 1)),
    ((3, 4, 2), 6, (1, 0, 0, 0, 0, 1)),
    ((3, 2, 3), 7, (0, 0, 1, 1, 0, 0)),
]


@pytest.mark.parametrize("m,k,bc", CASES)
def test_fe_box_operator_matches_oracle_for_every_brick(m, k, bc):
    from paper_1910_01900_gb300 import Context
    from paper_1910_01900_gb300.csrc_info import max_cells_per_block
    lo, hi = (0.0, -0.5, 0.25), (1.0, 1.0, 1.0)
    ctx = Context(m, k, lo=lo, hi=hi, bc=bc, fe_assemble=0, lambda_override=2.0)
    level = ctx.num_levels - 2
    u = sipg_inputs.uniform(ctx.num_dofs(level), 50 + k)
    ref = FESpace(Mesh(m, lo=lo, hi=hi, bc=bc), k).apply(u)
    for dt, prec, tol in ((torch.float64, 0, 1e-12), (torch.float32, 1, 1e-5)):
        ug = torch.as_tensor(u).cuda().to(dt)
        first = None
        for cb in (0, 1, 8, 27):
            if cb > max_cells_per_block(k + 1, 8 >> prec):
                continue
            ctx.set_tile_shape(prec, 2, cb, level=level)
            v = torch.full_like(ug, float("nan"))
            ctx.level_apply(level, ug, v)
            torch.cuda.synchronize()
            if first is None:
                first = v
                assert close(v.cpu().numpy().astype(np.float64), ref) <= tol
            assert torch.equal(v, first), (prec, cb)
