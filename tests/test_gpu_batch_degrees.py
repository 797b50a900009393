"""The batched operator, one launch per degree and pass, at every degree (GPU).

Each problem's result is the one its own launch gives, bit for bit: the same
bodies on the same cells.  Two problems of each degree, with cell counts that
leave a remainder in the last block and a single cell among them.
"""
import pytest

import sipg_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deform", [0, 1])
@pytest.mark.parametrize("on_stream", [False, True])
def test_batched_operator_equals_single_launches(deform, on_stream):
    from paper_1910_01900_gb300 import Batch
    probs = [dict(m=(3, 2, 3), k=k, deform=deform) for k in range(1, 9)]
    probs += [dict(m=(1, 1, 1) if k > 4 else (5, 4, 5), k=k, deform=deform) for k in range(1, 9)]
    s = torch.cuda.Stream() if on_stream else None
    B = Batch(probs, stream=s)
    us = [torch.as_tensor(sipg_inputs.uniform(B.num_dofs(i), 60 + i)).cuda() for i in range(len(probs))]
    vs = [torch.full_like(u, float("nan")) for u in us]
    torch.cuda.synchronize()
    B.apply(us, vs)
    torch.cuda.synchronize()
    for i, u in enumerate(us):
        v = torch.empty_like(u)
        B.contexts[i].apply(u, v)
        torch.cuda.synchronize()
        assert torch.equal(v, vs[i]), probs[i]
