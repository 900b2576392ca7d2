"""The backward's causal mask: a query row that is not a number leaves dV of the keys it does not see as it was, bit for bit (its masked
probabilities are exactly 0 whatever its logsumexp is)."""
import math

import pytest

pytestmark = pytest.mark.gpu


# rows in the middle of a tile, at its ends and next to a ragged end; one CTA per key tile, shared key tiles and every kernel by head dimension
@pytest.mark.parametrize("B,Hq,n,d,row", [(1, 2, 128, 64, 63), (1, 8, 300, 64, 128), (1, 2, 200, 128, 127), (2, 16, 513, 128, 300),
                                          (1, 4, 257, 96, 200), (1, 2, 300, 192, 129), (1, 2, 190, 256, 64)])
def test_a_bad_query_row_reaches_no_key_behind_it(B, Hq, n, d, row):
    import torch
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build as mbuild
    mbuild.build()
    gen = torch.Generator(device="cuda").manual_seed(n + d)
    Q, K, V, dO = (torch.randn(B, Hq, n, d, generator=gen, device="cuda").bfloat16() for _ in range(4))
    desc = mb.make_desc(B, Hq, n, d, True, 1.0 / math.sqrt(d))
    ws = torch.empty(mb.moa_attn_workspace_bytes(desc, mb.MOA_OP_FUSED), dtype=torch.uint8, device="cuda")

    def dv(q):
        O, dQ, dK, dV = (torch.empty_like(Q) for _ in range(4))
        L = torch.empty(B, Hq, n, device="cuda")
        mb.moa_attn_fused_fwd_bwd(desc, q, K, V, dO, O, L, dQ, dK, dV, ws)
        torch.cuda.synchronize()
        assert mb.moa_last_device_status() == 0
        return dV

    bad = Q.clone()
    bad[:, :, row] = float("nan")
    good, other = dv(Q), dv(bad)
    assert torch.equal(good[:, :, row + 1:], other[:, :, row + 1:])
    assert torch.isnan(other[:, :, :row + 1]).any()
