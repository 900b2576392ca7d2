"""Decode on clusters of every size, also those that are no power of two, and through memory in one and two rounds: single heads, pairs and the
ring kernel's larger groups.  The number of launches tells a cluster (one) from a merge through memory (two)."""
import math

import numpy as np
import pytest

import oracle
from paper_2609_33916_b200 import inputs as mi
from test_decode_gpu import _inputs, _run, rt  # noqa: F401

pytestmark = pytest.mark.gpu

# on 148 SMs: segments 3, 6, 7 | ring: 1, 2, 3, 5, 6, 8, 2 | 18, 9, 74 through memory in one round, 12 in two
CASES = [("bf16", 75, 2, 2, 3001, 128, 1), ("bf16", 5, 16, 8, 1999, 128, 1), ("bf16", 37, 2, 1, 3001, 64, 1),
         ("f32", 13, 32, 8, 300, 128, 1), ("f32", 19, 32, 8, 2100, 64, 1), ("f32", 5, 32, 8, 900, 64, 1), ("f32", 3, 32, 8, 1537, 128, 1),
         ("f32", 11, 8, 2, 1700, 64, 1), ("f32", 15, 4, 1, 2500, 64, 1), ("f32", 3, 40, 8, 1100, 64, 1),
         ("f32", 1, 32, 8, 6001, 64, 2), ("f32", 2, 32, 8, 9001, 64, 2), ("f32", 1, 5, 1, 40000, 64, 2), ("f32", 3, 32, 8, 40001, 64, 2)]


@pytest.mark.parametrize("dtype,B,H,Hkv,n,d,launches", CASES)
def test_segments(rt, dtype, B, H, Hkv, n, d, launches):  # noqa: F811
    from paper_2609_33916_b200 import binding as mb
    q, K, V = _inputs(B, H, Hkv, n, d, seed=n + H, dtype=dtype)
    before = mb.moa_launch_count()
    got, lse = _run(rt, q, K, V, 1.0 / math.sqrt(d), dtype)
    assert mb.moa_launch_count() - before == launches
    ref = oracle.decode_attn(*(mi.to_f64(t, dtype) for t in (q, K, V)), 1.0 / math.sqrt(d))
    assert np.all(np.isfinite(got)) and mi.rel_err(got, ref["o"]) <= (1e-2 if dtype == "bf16" else 1e-5)
    assert np.max(np.abs(lse - ref["lse"])) <= (1e-3 if dtype == "bf16" else 1e-4)
