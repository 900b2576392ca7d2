"""The forward at head dimensions 136..256: two warpgroups share one accumulator and hand the row maximum from key tile to key tile.
Scores that grow with the keys (every tile raises the maximum of many rows, by either warpgroup), one tile to many, ragged tails, empty
columns, shared K/V heads, alone and with the backward's inputs written by the forward."""
import math

import numpy as np
import pytest

import oracle
from paper_2609_33916_b200 import inputs as mi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import gpu_harness
    from paper_2609_33916_b200 import build as mbuild
    mbuild.build()
    return gpu_harness


CASES = [(1, 2, 2, 127, 136, False), (1, 2, 1, 129, 192, True), (2, 2, 2, 385, 200, False), (1, 4, 1, 640, 256, True),
         (1, 3, 3, 1100, 192, False), (2, 2, 2, 897, 256, False)]


@pytest.mark.parametrize("B,Hq,Hkv,n,d,causal", CASES)
@pytest.mark.parametrize("op,layout", [("fused", 0), ("split", 1), ("fwd", 0)])
def test_row_maximum_grows_from_tile_to_tile(H, B, Hq, Hkv, n, d, causal, op, layout):
    q = mi.make_inputs(B, Hq, n, d, 500 + n, "bf16")
    kv = mi.make_inputs(B, Hkv, n, d, 1500 + n, "bf16")
    grow = np.minimum(np.arange(n) // 128, 4).astype(np.uint16)[:, None]        # K times 2^grow: exact in bf16
    K = np.where(kv["K"] & 0x7F80, kv["K"] + (grow << 7), kv["K"]).astype(np.uint16)
    inp = {"Q": q["Q"], "dO": q["dO"], "K": K, "V": kv["V"]}
    scale = 1.0 / math.sqrt(d)
    got = H.run_library(inp, "bf16", causal, scale, op=op, layout=layout)
    f = H.f64_inputs(inp, "bf16")
    ref = oracle.attn_fwd_bwd_gqa(f["Q"], f["K"], f["V"], f["dO"], causal, scale)
    H.assert_close(got, ref, H.TOL_BF16, keys=("O",) if op == "fwd" else ("O", "dQ", "dK", "dV"), tag=f"H{Hq}/{Hkv} n{n} d{d} {op}")
    assert mi.rel_err(got["L"], ref["L"]) <= 1e-3


# two CTAs per query tile: the fewest key tiles, ragged ones, all that run at once and one head more; columns that fill half, most and all of the
# second half
@pytest.mark.parametrize("B,Hq,Hkv,n,d,causal", [(1, 2, 2, 265, 200, False), (1, 3, 1, 257, 256, True), (1, 4, 2, 700, 224, True), (2, 1, 1, 1000, 256, True), (1, 1, 1, 1409, 208, False),
                                                 (1, 18, 18, 500, 256, False), (1, 19, 19, 500, 256, False), (1, 8, 1, 1500, 240, True)])
@pytest.mark.parametrize("op,layout", [("fwd", 1), ("split", 0)])
def test_few_query_tiles(H, B, Hq, Hkv, n, d, causal, op, layout):
    test_row_maximum_grows_from_tile_to_tile(H, B, Hq, Hkv, n, d, causal, op, layout)
