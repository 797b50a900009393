"""The one-pass operator on axis-aligned cells against the oracle (GPU).

Its blocks take cells in pairs per direction, so the sizes that matter are a
single cell, odd numbers of cells (a cell without a partner) in every
direction, and all block shapes; each result is compared element by element
with the FP64 oracle (FP64 <= 1e-12, FP32 <= 1e-5, the bounds of the operator
parity tests) and bit for bit between block shapes.
"""
import numpy as np
import pytest

import sipg_inputs
from oracle.dg import SIPG
from oracle.mesh import Mesh
from parity_check import close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # cells, degree, boundary codes (0 Dirichlet, 1 Neumann)
    ((1, 1, 1), 1, (0, 0, 0, 0, 0, 0)),
    ((1, 1, 1), 8, (0, 1, 0, 0, 1, 0)),
    ((2, 3, 5), 2, (1, 0, 0, 1, 0, 0)),
    ((5, 2, 3), 3, (0, 1, 1, 0, 1, 0)),
    ((7, 1, 2), 4, (0, 0, 1, 1, 0, 0)),
    ((3, 5, 1), 5, (1, 1, 0, 0, 1, 1)),
    ((3, 3, 3), 6, (0, 0, 0, 1, 0, 1)),
    ((1, 4, 3), 7, (0, 1, 0, 1, 0, 1)),
    ((9, 2, 1), 1, (0, 1, 0, 0, 0, 0)),
]


@pytest.mark.parametrize("m,k,bc", CASES)
def test_box_operator_matches_oracle_for_every_block_shape(m, k, bc):
    from paper_1910_01900_gb300 import Context
    from paper_1910_01900_gb300.csrc_info import max_cells_per_block
    lo, hi = (0.0, -0.5, 0.25), (1.0, 1.0, 1.0)
    ctx = Context(m, k, lo=lo, hi=hi, bc=bc, operator_only=True)
    u = sipg_inputs.uniform(ctx.num_dofs(), 5 + k)
    ref = SIPG(Mesh(m, lo=lo, hi=hi, bc=bc), k).apply(u)
    for dt, prec, tol in ((torch.float64, 0, 1e-12), (torch.float32, 1, 1e-5)):
        ug = torch.as_tensor(u).cuda().to(dt)
        first = None
        mx = max_cells_per_block(k + 1, 8 >> prec)
        for cb in sorted({0, 1, 2, 4, 7, 8, 16, mx}):
            if cb > mx:
                continue
            ctx.set_tile_shape(prec, 1, cb)
            v = torch.full_like(ug, float("nan"))
            ctx.apply(ug, v)
            torch.cuda.synchronize()
            if first is None:
                first = v
                assert close(v.cpu().numpy().astype(np.float64), ref) <= tol
            assert torch.equal(v, first), (prec, cb)
