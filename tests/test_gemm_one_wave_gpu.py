"""Plain products on either side of the line between pairs of CTAs and single ones (the shapes whose tiles test_gemm_rule.py names), compared with a float64
product; and run with pairs forbidden and forced, which has to give the same bits: the order of the additions over K is that of the K blocks in
every form."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# M, N, K, storage of A and B, residual: all tiles at once or not; 48 blocks of K or 49; K-major rows of whole sectors or not; K past a block
SHAPES = [(4608, 1024, 2048, 0, 0, False), (4864, 1024, 2048, 0, 0, True), (4608, 1024, 3072, 0, 1, True), (4608, 1024, 3080, 0, 1, False),
          (2048, 2048, 3136, 1, 1, False), (4096, 1024, 1056, 0, 0, True), (4080, 1024, 1032, 0, 0, False), (1984, 1200, 2920, 0, 0, True),
          (5312, 768, 1800, 1, 0, False), (4096, 1024, 1040, 1, 0, True), (4096, 1024, 568, 0, 0, False), (4096, 1024, 584, 0, 0, False),
          (3072, 1024, 1300, 1, 1, False), (1024, 2728, 1300, 1, 1, True)]


def operands(torch, M, N, K, a, b, res):
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    R = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    return R(*((K, M) if a else (M, K))), R(*((K, N) if b else (N, K))), R(M, N) if res else None


def product(torch, mb, shape):
    M, N, K, a, b, res = shape
    A, B, r = operands(torch, *shape)
    C = torch.full((M, N), float("nan"), device="cuda").bfloat16()
    mb.moa_gemm(mb.make_gemm_desc(M, N, K, a, b), A, B, C, R=r)
    torch.cuda.synchronize()
    assert mb.moa_last_device_status() == 0
    return A, B, r, C


@pytest.mark.parametrize("shape", SHAPES)
def test_products_at_the_line(shape):
    import torch
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build as mbuild
    mbuild.build()
    A, B, r, C = product(torch, mb, shape)
    ref = (A.double().T if shape[3] else A.double()) @ (B.double() if shape[4] else B.double().T) + (r.double() if shape[5] else 0)
    # one bf16 rounding of the result: at most 2^-9 of each element, and so of the norm
    assert ((C.double() - ref).norm() / ref.norm()).item() <= 2.0 ** -9


def test_pairs_and_single_tiles_give_the_same_bits(tmp_path):
    import torch
    from paper_2609_33916_b200 import build as mbuild
    mbuild.build()
    out = {}
    for mode in ("0", "1", "2"):       # never pairs, by the rule, always pairs (read once by a process)
        path = str(tmp_path / mode)
        subprocess.run([sys.executable, os.path.abspath(__file__), path], check=True, timeout=300,
                       env=dict(os.environ, MOA_GEMM_PAIR=mode, PYTHONPATH=mbuild.ROOT))
        out[mode] = torch.load(path)
    for i, shape in enumerate(SHAPES):
        assert torch.equal(out["0"][i], out["2"][i]) and torch.equal(out["1"][i], out["2"][i]), shape


if __name__ == "__main__":
    import torch
    from paper_2609_33916_b200 import binding as mb
    torch.save([product(torch, mb, s)[3].cpu() for s in SHAPES], sys.argv[1])
