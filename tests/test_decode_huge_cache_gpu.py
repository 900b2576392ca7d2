"""Grouped decode over one cache of 18 GB: the bytes that decide between a cluster and every SM do not fit an int."""
import pytest

pytestmark = pytest.mark.gpu


def test_every_sm_takes_part():
    torch = pytest.importorskip("torch")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    build.build()
    n, d, H = 35_600_001, 128, 4
    if torch.cuda.mem_get_info()[0] < 24 << 30:
        pytest.skip("needs 24 GB of free memory")
    K = torch.zeros((1, 1, n, d), dtype=torch.bfloat16, device="cuda")
    V = torch.ones((1, 1, n, d), dtype=torch.bfloat16, device="cuda")
    V[:, :, -1] = float(n)      # (the last, ragged tile counts)
    q = torch.randn((1, H, d), device="cuda").bfloat16()
    out = torch.empty_like(q)
    lse = torch.empty((1, H), dtype=torch.float32, device="cuda")
    desc = mb.make_decode_desc(1, H, n, d, 0.1, H_kv=1)
    ws = torch.empty(mb.moa_decode_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    before = mb.moa_launch_count()
    mb.moa_decode_attn(desc, q, K, V, out, lse, ws)
    launches = mb.moa_launch_count() - before
    assert mb.moa_last_device_status() == mb.MOA_OK
    # every weight is 1 / n: one rounding of n to bf16 in V, one of the result, and fp32 sums of 35.6M ones over 148 x 8 warps, each exact
    want = (n - 1 + float(torch.tensor(float(n)).bfloat16())) / n
    assert (out.double() - want).abs().max().item() <= 2 ** -8 * want
    assert (lse.double() - torch.log(torch.tensor(float(n), dtype=torch.float64))).abs().max().item() <= 1e-5
    assert launches == 2      # all SMs and a merge, not one cluster of eight CTAs
    del K, V
    torch.cuda.empty_cache()
