"""Forward calls of so few work items that each CTA has at most one: items of one Q tile instead of two."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_07524_b200 import binding as B
from paper_2608_07524_b200 import inputs

pytestmark = pytest.mark.gpu


def forward(lengths, H, d, causal, heads=None):
    """(o, lse, the inputs on the host); `heads`: how many of the H heads the call is given."""
    cu = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int32)
    T = int(cu[-1])
    q, k, v, _ = inputs.make_qkvg(T, H, d, 40 + H)
    n = heads or H
    qd, kd, vd = (x[:, :n].contiguous().cuda() for x in (q, k, v))
    ws = B.alloc_workspace(T, len(lengths), n, d, False, "cuda")
    o, lse = B.dcp_varlen_attn_fwd(qd, kd, vd, torch.tensor(cu, device="cuda"), max(lengths), causal, workspace=ws)
    B.dcp_query_status(ws)
    return o, lse, (q, k, v, cu)


@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("d", [64, 72, 96, 112, 128])
@pytest.mark.parametrize("lengths", [[129], [128, 256, 257], [385, 1, 0, 640], [13, 40, 128, 500]], ids=lambda x: "-".join(map(str, x)))
def test_one_tile_items(lengths, d, causal):
    """Against the oracle (its tolerances: bf16 operands and results), and the same bits as in a call of many heads, whose
    items are two tiles: a tile's sums do not depend on what shares its item."""
    n_sms = torch.cuda.get_device_properties(0).multi_processor_count
    few = 2
    assert (sum(lengths) // 128 + len(lengths)) * few <= n_sms
    many = n_sms // (sum(lengths) // 128 + len(lengths)) + 1
    o, lse, (q, k, v, cu) = forward(lengths, many, d, causal, heads=few)
    O, L = oracle.attn_fwd(q[:, :few].contiguous(), k[:, :few].contiguous(), v[:, :few].contiguous(), cu, causal)
    got = o.double().cpu().numpy()
    assert np.max(np.abs(got - O)) <= 5e-2 and np.linalg.norm(got - O) <= 1e-2 * np.linalg.norm(O)
    assert np.max(np.abs(lse.double().cpu().numpy() - L)) <= 2e-3
    o2, lse2, _ = forward(lengths, many, d, causal)
    assert torch.equal(o, o2[:, :few]) and torch.equal(lse, lse2[:few])
