"""Decode without grouping where the number of cache segments changes: heads that just fit the GPU in clusters of 8, 4 and 2 and one more,
the last count that is merged through memory and the first that is not, few keys per segment, pairs of heads, and several waves."""
import math

import numpy as np
import pytest

import oracle
from paper_2609_33916_b200 import inputs as mi
from test_decode_gpu import _inputs, _run, rt  # noqa: F401

pytestmark = pytest.mark.gpu


def _check(got, lse, ref, dtype):
    assert np.all(np.isfinite(got)) and mi.rel_err(got, ref["o"]) <= (1e-2 if dtype == "bf16" else 1e-5)
    assert np.max(np.abs(lse - ref["lse"])) <= (1e-3 if dtype == "bf16" else 1e-5)


@pytest.mark.parametrize("B,H,Hkv,n,d,dtype", [
    (37, 2, 2, 1100, 64, "bf16"), (25, 3, 3, 1100, 64, "bf16"), (37, 4, 4, 1025, 128, "f32"), (149, 1, 1, 640, 64, "f32"),
    (37, 8, 8, 513, 64, "bf16"), (27, 11, 11, 300, 64, "f32"), (37, 1, 1, 5600, 64, "bf16"), (38, 1, 1, 5600, 64, "bf16"),
    (37, 1, 1, 5400, 64, "bf16"), (1, 5, 5, 513, 64, "f32"), (1, 5, 5, 512, 64, "f32"), (1, 5, 5, 129, 128, "bf16"),
    (55, 2, 1, 1100, 64, "bf16"), (56, 2, 1, 1100, 64, "bf16"), (27, 2, 1, 6000, 64, "f32")])
def test_edges_of_the_segment_rule(rt, B, H, Hkv, n, d, dtype):  # noqa: F811
    q, K, V = _inputs(B, H, Hkv, n, d, seed=n + B, dtype=dtype)
    got, lse = _run(rt, q, K, V, 1.0 / math.sqrt(d), dtype)
    ref = oracle.decode_attn(*(mi.to_f64(t, dtype) for t in (q, K, V)), 1.0 / math.sqrt(d))
    _check(got, lse, ref, dtype)


@pytest.mark.parametrize("B,n", [(19, 15800), (40, 7900)])
def test_long_segments_in_several_waves(rt, B, n):  # noqa: F811
    """152 and 320 heads of 500 KB segments; the batch entries have the same cache and their own query."""
    q, K, V = _inputs(1, 8, 8, n, 64, seed=n, dtype="bf16")
    qs = _inputs(B, 8, 8, 1, 64, seed=B, dtype="bf16")[0]
    got, lse = _run(rt, qs, np.repeat(K, B, 0), np.repeat(V, B, 0), 0.125, "bf16")
    for b in range(0, B, 6):
        ref = oracle.decode_attn(*(mi.to_f64(t, "bf16") for t in (qs[b:b + 1], K, V)), 0.125)
        _check(got[b:b + 1], lse[b:b + 1], ref, "bf16")
