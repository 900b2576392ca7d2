"""The register-tiled CUDA-core kernels at the edges of their tiles and of the rule that picks them: 2, 4 or 8 rows per
thread (the fewer the smaller the problem), one CTA or a cluster of 2, 4, 8 per output tile, ragged tails of both axes."""
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


# B, H, n, d: two rows per thread with and without a second key tile | four rows | eight, in clusters of 4, 2 and alone |
# the 128-column kernels: two and four rows, clusters and alone
CASES = [(1, 1, 16, 64), (1, 1, 17, 64), (1, 2, 129, 64), (1, 4, 300, 64), (1, 1, 511, 64), (1, 16, 193, 64), (2, 33, 129, 64),
         (2, 96, 128, 64), (1, 1, 31, 128), (1, 1, 289, 128), (1, 8, 225, 128), (1, 40, 97, 128), (2, 64, 96, 128)]


@pytest.mark.parametrize("op", ["fused", "split"])
@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("B,Hh,n,d", CASES)
def test_fp32_tile_edges(H, B, Hh, n, d, causal, op):
    inp = mi.make_inputs(B, Hh, n, d, seed=900 + n, dtype="f32")
    scale = 1.0 / math.sqrt(d)
    ref = oracle.attn_fwd_bwd(*(mi.to_f64(inp[k], "f32") for k in ("Q", "K", "V", "dO")), causal, scale)
    got = H.run_library(inp, "f32", causal, scale, op=op)
    H.assert_close(got, ref, H.TOL_F32, keys=("O", "L", "dQ", "dK", "dV"), tag=f"B{B} H{Hh} n{n} d{d}")


@pytest.mark.parametrize("op", ["fused", "split"])
@pytest.mark.parametrize("n,d,scale", [(65, 64, 0.125), (130, 64, -0.125), (97, 128, 0.09)])
def test_bf16_storage_on_the_cuda_cores(H, n, d, scale, op):
    inp = mi.make_inputs(1, 3, n, d, seed=950 + n, dtype="bf16")
    ref = oracle.attn_fwd_bwd(*(mi.to_f64(inp[k], "bf16") for k in ("Q", "K", "V", "dO")), True, scale)
    got = H.run_library(inp, "bf16", True, scale, op=op, path=mb.MOA_PATH_SIMT)
    H.assert_close(got, ref, H.TOL_BF16, tag=f"n{n} d{d} scale{scale}")
