"""Decode at the edges of the rules that split the cache: one CTA, clusters of 2, 4 and 8 (some with empty segments), more
segments than a cluster holds (merged through the workspace), small and large groups of query heads."""
import math

import numpy as np
import pytest

import oracle
from paper_2609_33916_b200 import inputs as mi
from test_decode_gpu import _inputs, _run, rt  # noqa: F401

pytestmark = pytest.mark.gpu

CASES = [(1, 1, 1, 128, 64), (1, 1, 1, 129, 64), (2, 2, 2, 385, 128), (1, 2, 2, 1024, 64), (1, 2, 1, 1025, 64), (3, 50, 50, 513, 64),
         (1, 3, 1, 700, 128), (5, 6, 3, 2048, 64), (40, 16, 16, 131, 128),
         # groups of 4 to 16: fewer units than SMs, heads shared by several CTAs, several heads per CTA, one partial tile
         (1, 8, 1, 900, 64), (2, 32, 4, 300, 128), (1, 4, 1, 1, 128), (1, 5, 1, 63, 64), (40, 32, 8, 65, 128), (3, 32, 2, 5000, 128),
         (2, 13, 1, 20000, 64), (1, 16, 1, 9473, 128)]


@pytest.mark.parametrize("dtype,tol", [("bf16", 1e-2), ("f32", 1e-5)])
@pytest.mark.parametrize("B,H,Hkv,n,d", CASES)
def test_decode_splits(rt, dtype, tol, B, H, Hkv, n, d):  # noqa: F811
    q, K, V = _inputs(B, H, Hkv, n, d, seed=n + H, dtype=dtype)
    got, lse = _run(rt, q, K, V, 1.0 / math.sqrt(d), dtype)
    ref = oracle.decode_attn(mi.to_f64(q, dtype), mi.to_f64(K, dtype), mi.to_f64(V, dtype), 1.0 / math.sqrt(d))
    assert np.all(np.isfinite(got)) and mi.rel_err(got, ref["o"]) <= tol
    assert np.max(np.abs(lse - ref["lse"])) <= (1e-3 if dtype == "bf16" else 1e-4)
