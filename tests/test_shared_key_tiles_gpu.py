"""The backward with several CTAs per key tile (a cluster shares the tile's query tiles and adds the partial dK, dV): shapes with
few key tiles, for every cluster size, group size and head dimension, parts that are empty or cross from one query head to the
next, ragged tails, both fixed layouts."""
import math

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


CASES = [
    # B, H, H_kv, n, d, causal
    (1, 1, 1, 129, 128, True),        # the last key tile has one query tile: a part without any
    (1, 1, 1, 1100, 64, False),
    (1, 2, 2, 1030, 128, False),
    (1, 3, 3, 1500, 128, True),
    (2, 8, 2, 300, 128, True),
    (1, 6, 1, 450, 64, True),         # parts begin in the middle of a query head
    (1, 16, 1, 257, 80, False),
    (1, 1, 1, 130, 192, True),
    (1, 6, 2, 333, 256, False),
    (1, 16, 4, 500, 192, True),
]


@pytest.mark.parametrize("B,Hq,Hkv,n,d,causal", CASES)
@pytest.mark.parametrize("op,layout", [("fused", 0), ("split", 1)])
def test_shared_key_tiles(H, B, Hq, Hkv, n, d, causal, op, layout):
    q = mi.make_inputs(B, Hq, n, d, 700 + n, "bf16")
    kv = mi.make_inputs(B, Hkv, n, d, 1700 + n, "bf16")
    inp = {"Q": q["Q"], "dO": q["dO"], "K": kv["K"], "V": kv["V"]}
    scale = 1.0 / math.sqrt(d)
    got = H.run_library(inp, "bf16", causal, scale, op=op, layout=layout)
    f = H.f64_inputs(inp, "bf16")
    ref = oracle.attn_fwd_bwd_gqa(f["Q"], f["K"], f["V"], f["dO"], causal, scale)
    H.assert_close(got, ref, H.TOL_BF16, tag=f"H{Hq}/{Hkv} n{n} d{d}")


@pytest.mark.parametrize("B,Hq,Hkv,n,d,causal", [(2, 40, 40, 64, 136, False), (2, 40, 40, 65, 192, True), (3, 60, 60, 200, 160, True),
                                                 (2, 80, 40, 129, 192, False), (1, 160, 160, 128, 184, True), (1, 8, 1, 700, 192, False),
                                                 (1, 3, 3, 1000, 144, True)])
@pytest.mark.parametrize("op,dq_mode,layout", [("fused", 0, 0), ("split", 1, 1)])
def test_one_pass_backward_up_to_192(H, B, Hq, Hkv, n, d, causal, op, dq_mode, layout):
    """136..192 columns: one and several CTAs per key tile, one and many query tiles, every number of columns in the last box."""
    q = mi.make_inputs(B, Hq, n, d, 800 + n, "bf16")
    kv = mi.make_inputs(B, Hkv, n, d, 1800 + n, "bf16")
    inp = {"Q": q["Q"], "dO": q["dO"], "K": kv["K"], "V": kv["V"]}
    scale = 1.0 / math.sqrt(d)
    got = H.run_library(inp, "bf16", causal, scale, op=op, layout=layout, dq_mode=dq_mode)
    f = H.f64_inputs(inp, "bf16")
    ref = oracle.attn_fwd_bwd_gqa(f["Q"], f["K"], f["V"], f["dO"], causal, scale)
    H.assert_close(got, ref, H.TOL_BF16, tag=f"H{Hq}/{Hkv} n{n} d{d}")
