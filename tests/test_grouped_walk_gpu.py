"""dQ of several query heads that share a K/V head, sent by add-reduces of 128 columns: the (query head, tile) each of them goes to, for one CTA per
key tile and for parts of a walk that begin and end inside a head, one and many tiles per head, ragged tails."""
import math

import pytest

import oracle
from paper_2609_33916_b200 import binding as mb
from paper_2609_33916_b200 import inputs as mi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import gpu_harness
    from paper_2609_33916_b200 import build as mbuild
    mbuild.build()
    return gpu_harness


# the mode a caller names keeps one CTA per key tile; the default one shares key tiles where there are few
@pytest.mark.parametrize("mode", [mb.MOA_DQ_AUTO, mb.MOA_DQ_BULK_REDUCE])
@pytest.mark.parametrize("B,Hq,Hkv,n,d,causal", [(1, 8, 1, 100, 128, True), (1, 8, 1, 129, 128, True), (1, 5, 1, 385, 128, False), (2, 6, 2, 500, 96, True),
                                                 (1, 12, 4, 257, 72, False), (1, 7, 1, 640, 104, True)])
def test_every_tile_of_the_walk(H, B, Hq, Hkv, n, d, causal, mode):
    q, kv = mi.make_inputs(B, Hq, n, d, 900 + n, "bf16"), mi.make_inputs(B, Hkv, n, d, 1900 + n, "bf16")
    inp = {"Q": q["Q"], "dO": q["dO"], "K": kv["K"], "V": kv["V"]}
    scale = 1.0 / math.sqrt(d)
    got = H.run_library(inp, "bf16", causal, scale, dq_mode=mode)
    f = H.f64_inputs(inp, "bf16")
    ref = oracle.attn_fwd_bwd_gqa(f["Q"], f["K"], f["V"], f["dO"], causal, scale)
    H.assert_close(got, ref, H.TOL_BF16, tag=f"H{Hq}/{Hkv} n{n} d{d}")
    # a tile sent to another head's or tile's rows would leave those of its own without their largest terms: each block of 128 rows by itself
    for h in range(Hq):
        for r in range(0, n, 128):
            a, b = got["dQ"][:, h, r:r + 128], ref["dQ"][:, h, r:r + 128]
            assert abs(a - b).max() <= H.TOL_BF16 * abs(ref["dQ"]).max(), (h, r)
