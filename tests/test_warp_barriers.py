"""Aligned barriers in hand-written instructions are undefined for a warp whose lanes arrive apart: every one of them stands right behind a
__syncwarp().  The merges of the fp32 kernels' clusters are where lanes do leave a loop apart: odd numbers of rows per rank at 64 columns
(two rows to a warp), and a ragged last tile."""
import glob
import math
import os
import re

import pytest

import oracle
from paper_2609_33916_b200 import build
from paper_2609_33916_b200 import inputs as mi


def test_aligned_barriers_behind_a_converged_warp():
    seen = 0
    for path in sorted(glob.glob(os.path.join(build.CSRC, "*.cu*"))):
        with open(path) as f:
            lines = f.read().split("\n")
        for i, line in enumerate(lines):
            if re.search(r"asm.*\"[^\"]*\bbar(rier)?\.(sync|arrive|cluster)", line):
                seen += 1
                assert lines[i - 1].strip() == "__syncwarp();", f"{os.path.basename(path)}:{i + 1}"
    assert seen >= 2


# B, H, n, d, causal: rows per rank of the forward (and of the backward) 13, 7, 3, 11, 10 and 5, the last rank with fewer; the last key tile
# ends inside a warp's pair of rows
@pytest.mark.gpu
@pytest.mark.parametrize("op", ["fused", "split"])
@pytest.mark.parametrize("B,Hh,n,d,causal", [(1, 2, 583, 64, False), (1, 1, 583, 64, False), (1, 1, 331, 64, False), (2, 1, 657, 64, False),
                                             (1, 1, 1175, 64, False), (1, 3, 399, 64, False), (1, 1, 1175, 64, True), (1, 1, 805, 128, False)])
def test_merges_of_odd_shares(B, Hh, n, d, causal, op):
    import gpu_harness as H
    build.build()
    inp = mi.make_inputs(B, Hh, n, d, seed=970 + n, dtype="f32")
    scale = 1.0 / math.sqrt(d)
    ref = oracle.attn_fwd_bwd(*(mi.to_f64(inp[k], "f32") for k in ("Q", "K", "V", "dO")), causal, scale)
    got = H.run_library(inp, "f32", causal, scale, op=op)
    H.assert_close(got, ref, H.TOL_F32, keys=("O", "L", "dQ", "dK", "dV"), tag=f"B{B} H{Hh} n{n} d{d}")
