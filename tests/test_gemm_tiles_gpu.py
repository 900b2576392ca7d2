"""Products at the edges of the rule that picks the tile: 64, 128 and 256 columns on single CTAs and pairs, tails in every
direction, against a float64 product of the same bf16 operands."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    build.build()
    return torch, mb


# M, N, K: one tile | a tail of one chunk | 64 columns, several rows | 128 columns | a pair of CTAs | 256 columns on single CTAs
SHAPES = [(8, 8, 8), (128, 72, 64), (136, 200, 520), (520, 640, 4096), (1704, 1000, 1024), (2048, 2304, 512), (104, 76808, 64)]


@pytest.mark.parametrize("a_layout,b_layout", [(0, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("res", [False, True])
def test_products(rt, M, N, K, a_layout, b_layout, res):
    torch, mb = rt
    gen = torch.Generator(device="cuda").manual_seed(M + N + K)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    A, B = (R(K, M) if a_layout else R(M, K)), (R(K, N) if b_layout else R(N, K)) * K ** -0.5
    add = R(M, N) if res else None
    C = torch.full((M, N), float("nan"), device="cuda", dtype=torch.bfloat16)
    mb.moa_gemm(mb.make_gemm_desc(M, N, K, a_layout, b_layout), A, B, C, R=add)
    assert mb.moa_last_device_status() == mb.MOA_OK
    ref = (A.double().T if a_layout else A.double()) @ (B.double() if b_layout else B.double().T)
    if res:
        ref = ref + add.double()
    # one rounding to bf16 of the result (2^-9 of an element), fp32 sums far below that
    assert (C.double() - ref).abs().max().item() <= 2 ** -8 * ref.abs().max().item()


@pytest.mark.parametrize("n,d,dff", [(8, 64, 72), (300, 128, 1000), (700, 1024, 648), (2100, 256, 2048)])
def test_gated_mlp_widths(rt, n, d, dff):
    torch, mb = rt
    gen = torch.Generator(device="cuda").manual_seed(n)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    x, W1, W3, W2, dy = R(n, d), R(dff, d) * d ** -0.5, R(dff, d) * d ** -0.5, R(d, dff) * dff ** -0.5, R(n, d)
    E = lambda *s: torch.full(s, float("nan"), device="cuda", dtype=torch.bfloat16)      # noqa: E731
    a, u, h, y, dx, dW1, dW3, dW2 = E(n, dff), E(n, dff), E(n, dff), E(n, d), E(n, d), E(dff, d), E(dff, d), E(d, dff)
    desc = mb.make_mlp_desc(n, d, dff)
    ws = torch.empty(mb.moa_gated_mlp_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    mb.moa_gated_mlp_fwd(desc, x, W1, W3, W2, a, u, h, y)
    mb.moa_gated_mlp_bwd(desc, x, W1, W3, W2, a, u, h, dy, dx, dW1, dW3, dW2, ws)
    assert mb.moa_last_device_status() == mb.MOA_OK
    f = lambda t: t.double()                                                     # noqa: E731
    ra, ru = f(x) @ f(W1).T, f(x) @ f(W3).T
    rh = torch.nn.functional.silu(ra) * ru
    # the backward from the a, u, h that were stored (bf16), as the library has them
    sa, su = f(a), f(u)
    s = torch.sigmoid(sa)
    dh = f(dy) @ f(W2)
    da, du = dh * su * s * (1 + sa * (1 - s)), dh * sa * s
    for got, ref in ((a, ra), (u, ru), (h, rh), (y, f(h) @ f(W2).T), (dW2, f(dy).T @ f(h)), (dW1, da.T @ f(x)), (dW3, du.T @ f(x)),
                     (dx, da @ f(W1) + du @ f(W3))):
        assert (got.double() - ref).abs().max().item() <= 1e-2 * ref.abs().max().item()


@pytest.mark.parametrize("B,n,H,d,dff", [(1, 40, 1, 64, 72), (2, 186, 4, 128, 1360), (1, 700, 8, 64, 1024), (1, 1613, 16, 64, 1000)])
def test_block_products_side_by_side(rt, B, n, H, d, dff):
    """The products a block's backward may launch together.  dWo against the block's three-projection form, where it is a launch of its own, bit
    for bit; dx and what comes from dqkv up to the atomics in dQ.  (The MLP's four products are launched together, or not, in both forms alike:
    test_mlp_products_side_by_side.)"""
    torch, mb = rt
    from paper_2609_33916_b200.block import TransformerBlock
    gen = torch.Generator(device="cuda").manual_seed(n)
    dm = H * d
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    w = {k: R(dm, dm) * dm ** -0.5 for k in ("Wq", "Wk", "Wv", "Wo")}
    w.update(W1=R(dff, dm) * dm ** -0.5, W3=R(dff, dm) * dm ** -0.5, W2=R(dm, dff) * dff ** -0.5, g1=1 + 0.25 * R(dm), g2=1 + 0.25 * R(dm))
    x, dy = R(B * n, dm), R(B * n, dm)
    out = []
    for packed in (True, False):
        blk = TransformerBlock(torch, B, n, H, d, dff, True, packed_qkv=packed)
        wp = blk.prepare_weights(w)
        blk.forward(x, wp)
        dx, g = blk.backward(x, wp, dy)
        assert mb.moa_last_device_status() == mb.MOA_OK
        out.append({"y": blk.y.double(), "dx": dx.double(), **{k: v.double() for k, v in g.items()}})
    for k in ("y", "W1", "W2", "W3", "g2", "Wo"):
        assert torch.equal(out[0][k], out[1][k]), k
    for k in ("dx", "Wq", "Wk", "Wv", "g1"):      # bf16 results of dQ sums in another order (and dh1 as one sum of three)
        assert (out[0][k] - out[1][k]).abs().max().item() <= 1.6e-2 * out[1][k].abs().max().item(), k


# 64-column tiles of all four products within a wave, 128-column tiles within one, and neither; tails of rows, columns and of the K loop
@pytest.mark.parametrize("n,d,dff,launches", [(40, 64, 72, 2), (700, 128, 264, 2), (520, 512, 1000, 2), (700, 1024, 1032, 4)])
def test_mlp_products_side_by_side(rt, n, d, dff, launches):
    """dW2, dW1, dW3 and dx of a gated MLP's backward against the same products one by one, from the da, du that the call left in its workspace:
    one fp32 accumulation over K in the same order whichever tile or launch, so the same bits (dx: two sums instead of one of both)."""
    torch, mb = rt
    gen = torch.Generator(device="cuda").manual_seed(n + dff)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    x, W1, W3, W2, dy = R(n, d), R(dff, d) * d ** -0.5, R(dff, d) * d ** -0.5, R(d, dff) * dff ** -0.5, R(n, d)
    a, u, h = R(n, dff), R(n, dff), R(n, dff)
    E = lambda *s: torch.full(s, float("nan"), device="cuda", dtype=torch.bfloat16)      # noqa: E731
    dx, dW1, dW3, dW2 = E(n, d), E(dff, d), E(dff, d), E(d, dff)
    desc = mb.make_mlp_desc(n, d, dff)
    ws = torch.empty(mb.moa_gated_mlp_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    before = mb.moa_launch_count()
    mb.moa_gated_mlp_bwd(desc, x, W1, W3, W2, a, u, h, dy, dx, dW1, dW3, dW2, ws)
    assert mb.moa_launch_count() - before == launches
    half = ws.numel() // 2
    da, du = (ws[i * half:i * half + 2 * n * dff].view(torch.bfloat16).view(n, dff) for i in range(2))
    f = lambda t: t.double()                                                     # noqa: E731
    s = torch.sigmoid(f(a))
    dh = f(dy) @ f(W2)
    for got, ref in ((da, dh * f(u) * s * (1 + f(a) * (1 - s))), (du, dh * f(a) * s)):
        assert (f(got) - ref).abs().max().item() <= 2 ** -7 * ref.abs().max().item()      # one rounding to bf16, a fast sigmoid below it

    def product(M, N, K, A, B, a_layout, b_layout, add=None):
        C = E(M, N)
        mb.moa_gemm(mb.make_gemm_desc(M, N, K, a_layout, b_layout), A, B, C, R=add)
        return C
    for name, got, A, B, M, N in (("dW2", dW2, dy, h, d, dff), ("dW1", dW1, da, x, dff, d), ("dW3", dW3, du, x, dff, d)):
        assert torch.equal(got, product(M, N, n, A, B, 1, 1)), name
    ref = f(da) @ f(W1) + f(du) @ f(W3)
    assert (f(dx) - ref).abs().max().item() <= 2 ** -8 * ref.abs().max().item()
    assert mb.moa_last_device_status() == mb.MOA_OK
