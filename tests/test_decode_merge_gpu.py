"""Grouped decode where a head is spread over many CTAs (one round of loads of the merge, several, and one CTA more than a round), where its
clusters stop fitting, and at the edges of the 128-key tiles of 64-column heads."""
import math

import numpy as np
import pytest

import oracle
from paper_2609_33916_b200 import inputs as mi
from test_decode_gpu import _inputs, _run, rt  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,H,Hkv,n,d", [(1, 8, 1, 20000, 64), (1, 16, 1, 30001, 128), (1, 32, 4, 16000, 64), (16, 8, 1, 5000, 64),
                                         (15, 4, 1, 4000, 128), (33, 4, 1, 2500, 64), (2, 12, 2, 127, 64), (1, 8, 2, 129, 64), (1, 16, 4, 257, 64)])
def test_many_ctas_per_head(rt, B, H, Hkv, n, d):  # noqa: F811
    q, K, V = _inputs(B, H, Hkv, n, d, seed=n + H, dtype="bf16")
    got, lse = _run(rt, q, K, V, 1.0 / math.sqrt(d), "bf16")
    ref = oracle.decode_attn(*(mi.to_f64(t, "bf16") for t in (q, K, V)), 1.0 / math.sqrt(d))
    assert np.all(np.isfinite(got)) and mi.rel_err(got, ref["o"]) <= 1e-2
    assert np.max(np.abs(lse - ref["lse"])) <= 1e-3
