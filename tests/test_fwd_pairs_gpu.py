"""The forward on pairs of query tiles: enough heads that it is chosen, odd and even numbers of query tiles, ragged last tiles,
shared K/V heads, head dimensions with empty columns, alone and inside the fused call."""
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


CASES = [(2, 75, 75, 256, 64, True), (2, 75, 75, 257, 64, False), (3, 64, 16, 300, 128, True), (2, 80, 80, 129, 96, False),
         (1, 160, 8, 384, 80, True), (1, 150, 150, 513, 128, False), (1, 100, 100, 640, 40, True), (1, 40, 40, 1100, 128, True)]


@pytest.mark.parametrize("B,Hq,Hkv,n,d,causal", CASES)
@pytest.mark.parametrize("op,layout", [("fused", 0), ("split", 1), ("fwd", 0)])
def test_query_tile_pairs(H, B, Hq, Hkv, n, d, causal, op, layout):
    q = mi.make_inputs(B, Hq, n, d, 300 + n, "bf16", gain=4.0)        # (scores wide enough for rescales)
    kv = mi.make_inputs(B, Hkv, n, d, 1300 + n, "bf16")
    inp = {"Q": q["Q"], "dO": q["dO"], "K": kv["K"], "V": kv["V"]}
    scale = 1.0 / math.sqrt(d)
    got = H.run_library(inp, "bf16", causal, scale, op=op, layout=layout)
    f = H.f64_inputs(inp, "bf16")
    ref = oracle.attn_fwd_bwd_gqa(f["Q"], f["K"], f["V"], f["dO"], causal, scale)
    H.assert_close(got, ref, H.TOL_BF16, keys=("O",) if op == "fwd" else ("O", "dQ", "dK", "dV"), tag=f"H{Hq}/{Hkv} n{n} d{d} {op}")
    assert mi.rel_err(got["L"], ref["L"]) <= 1e-3
