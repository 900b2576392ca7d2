"""The rule that cuts a product into tiles, on both sides of each of its lines (148 SMs): pairs of CTAs, single ones, narrower tiles.  The rule is plain
host arithmetic and is compiled by itself here; the products on either side are run by test_gemm_one_wave_gpu.py."""
import ctypes
import os
import subprocess

import pytest

from paper_2609_33916_b200 import build

SINGLE, PAIR = (256, False), (256, True)
SOURCE = """#include "gemm_rule.cuh"
extern "C" int tile(long long M, long long N, long long K, int a, int b, int plain, int dual, int two, int nbatch, long long sms, int mode)
{ const moa::GemmTile t = moa::gemm_tile(M, N, K, a, b, plain, dual, two, nbatch, sms, mode); return t.columns + (t.pair ? 1000 : 0); }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rule") / "rule.so")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-x", "c++", "-", "-o", so],
                   input=SOURCE, text=True, check=True)
    f = ctypes.CDLL(so).tile
    f.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 6 + [ctypes.c_longlong, ctypes.c_int]

    def tile(M, N, K, a=0, b=0, plain=1, dual=0, two=0, nbatch=1, sms=148, mode=1):
        t = f(M, N, K, a, b, plain, dual, two, nbatch, sms, mode)
        return t % 1000, t >= 1000
    return tile


# (a, b): the operand is stored by columns
@pytest.mark.parametrize("M,N,K,a,b,want", [
    # all single tiles at once (144), or not (152 in 76 pairs: two rounds either way)
    (4608, 1024, 2048, 0, 0, SINGLE), (4864, 1024, 2048, 0, 0, PAIR),
    # 48 blocks of K, or 49
    (4608, 1024, 3072, 0, 1, SINGLE), (4608, 1024, 3080, 0, 1, PAIR), (2048, 2048, 3072, 1, 1, SINGLE), (2048, 2048, 3136, 1, 1, PAIR),
    # K-major rows of 2 K bytes: whole 64 bytes, whole 32 bytes, neither
    (4096, 1024, 1024, 0, 0, SINGLE), (4096, 1024, 1056, 0, 0, SINGLE), (4080, 1024, 1040, 0, 0, PAIR), (4080, 1024, 1032, 0, 0, PAIR),
    (1984, 1200, 2920, 0, 0, PAIR), (4192, 720, 1976, 0, 0, PAIR), (3288, 808, 2632, 0, 0, PAIR),
    (5312, 768, 1800, 1, 0, PAIR), (4096, 1024, 1040, 1, 0, SINGLE), (4096, 1024, 1032, 0, 1, SINGLE),
    # ... over a short K
    (4096, 1024, 568, 0, 0, SINGLE), (4096, 1024, 584, 0, 0, PAIR), (4096, 1024, 816, 0, 0, SINGLE), (4096, 1024, 848, 0, 0, PAIR),
    # an operand stored by columns that does not come in by whole blocks of 64
    (1024, 2752, 1300, 1, 1, SINGLE), (1024, 2728, 1300, 1, 1, PAIR), (1032, 2752, 1300, 1, 1, PAIR)])
def test_one_wave(rule, M, N, K, a, b, want):
    assert rule(M, N, K, a, b) == want


def test_two_operand_pairs_count_both_loops(rule):
    assert rule(4608, 1024, 1536, 0, 1, two=1) == SINGLE and rule(4608, 1024, 1600, 0, 1, two=1) == PAIR
    assert rule(4608, 1024, 1600, 0, 1) == SINGLE


def test_gates_and_modes(rule):
    assert rule(4096, 512, 1024, plain=0, dual=1) == PAIR and rule(4096, 512, 1016, plain=0, dual=1)[1] is False
    for K in (1024, 1032, 3080):
        assert rule(4608, 1024, K, mode=2) == PAIR and rule(4608, 1024, K, mode=0)[1] is False


def test_narrow_tiles(rule):
    assert rule(512, 2048, 1024)[0] == 64 and rule(1024, 2048, 1024)[0] == 128 and rule(2048, 2048, 1024)[0] == 256
