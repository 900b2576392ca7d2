"""Plain products on either side of the line between pairs of CTAs and single ones: all tiles at once or one too many, K loops at the line."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,a_layout,b_layout,res", [
    (4736, 1024, 3072, 0, 0, False), (4737, 1024, 3072, 0, 0, True), (4736, 1024, 3073, 0, 1, False), (1300, 3072, 1000, 0, 0, True),
    (3072, 1024, 1300, 1, 1, False), (1024, 2728, 1300, 1, 1, False), (1300, 1024, 3200, 0, 1, True)])
def test_products_at_the_line(M, N, K, a_layout, b_layout, res):
    import torch
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build as mbuild
    mbuild.build()
    if (a_layout == 0 or b_layout == 0) and K % 8:
        K += 8 - K % 8            # (rows of K elements: 16 bytes)
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    R = lambda *s: torch.randn(*s, generator=gen, device="cuda").bfloat16()
    A, B, r = R(*((K, M) if a_layout else (M, K))), R(*((K, N) if b_layout else (N, K))), R(M, N)
    C = torch.full((M, N), float("nan"), device="cuda").bfloat16()
    mb.moa_gemm(mb.make_gemm_desc(M, N, K, a_layout, b_layout), A, B, C, R=r if res else None)
    torch.cuda.synchronize()
    assert mb.moa_last_device_status() == 0
    a, b = (A.double().T if a_layout else A.double()), (B.double() if b_layout else B.double().T)
    ref = a @ b + (r.double() if res else 0)
    # one bf16 rounding of the result: at most 2^-9 of each element, and so of the norm
    assert ((C.double() - ref).norm() / ref.norm()).item() <= 2.0 ** -9
