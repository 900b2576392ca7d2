"""Calls whose kernels start while their predecessors drain: chains of calls on reused buffers, behind a join of two
streams, under capture, give what the same calls give with a synchronisation after each."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    build.build()
    return torch, mb


def _chain(torch, mb, bufs, between):
    """fwd, bwd (dQ without atomics: bitwise reproducible), norm and product, each reading what the one before wrote."""
    B, H, n, d, x, w, g = bufs["shape"] + (bufs["x"], bufs["w"], bufs["g"])
    desc = mb.make_desc(B, H, n, d, True, 1.0 / math.sqrt(d), dq_mode=mb.MOA_DQ_SEPARATE_PASS)
    ws = bufs["ws"]
    E = lambda like: torch.empty_like(like)       # noqa: E731
    cur = x
    out = []
    for _ in range(3):
        O, dQ, dK, dV = E(cur), E(cur), E(cur), E(cur)
        L = torch.empty((B, H, n), dtype=torch.float32, device="cuda")
        mb.moa_attn_fwd(desc, cur, cur, cur, O, L); between()
        mb.moa_attn_bwd(desc, cur, cur, cur, O, L, O, dQ, dK, dV, ws); between()
        y, z = E(cur), E(cur)
        rows = B * H * n
        mb.moa_rmsnorm_fwd(mb.make_rmsnorm_desc(rows, d, 1e-5), dV, g, y); between()
        mb.moa_gemm(mb.make_gemm_desc(rows, d, d), y, w, z); between()
        cur = z
        out += [O, dQ, dK, dV, y, z]
    return out


@pytest.mark.parametrize("B,H,n,d", [(1, 2, 130, 64), (2, 4, 700, 128)])
def test_chains_of_calls(rt, B, H, n, d):
    torch, mb = rt
    gen = torch.Generator(device="cuda").manual_seed(n)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    desc = mb.make_desc(B, H, n, d, True, 1.0, dq_mode=mb.MOA_DQ_SEPARATE_PASS)
    bufs = {"shape": (B, H, n, d), "x": R(B, H, n, d), "w": R(d, d) * d ** -0.5, "g": R(d),
            "ws": torch.empty(mb.moa_attn_workspace_bytes(desc, mb.MOA_OP_BWD), dtype=torch.uint8, device="cuda")}
    ref = _chain(torch, mb, bufs, torch.cuda.synchronize)
    for _ in range(10):
        got = _chain(torch, mb, bufs, lambda: None)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, ref))


@pytest.mark.parametrize("captured", [False, True])
def test_call_behind_a_join_of_streams(rt, captured):
    """The call's inputs come from another stream: its first kernel has two predecessors."""
    torch, mb = rt
    B, H, n, d = 1, 4, 512, 128
    desc = mb.make_desc(B, H, n, d, False, 1.0 / math.sqrt(d))
    src = torch.randn(B, H, n, d, device="cuda").bfloat16()
    q, v, O = torch.zeros_like(src), torch.zeros_like(src), torch.zeros_like(src)
    big = torch.randn(4096, 4096, device="cuda")
    L = torch.empty((B, H, n), dtype=torch.float32, device="cuda")
    ref, Lr = torch.empty_like(src), torch.empty_like(L)
    mb.moa_attn_fwd(desc, src, src, src, ref, Lr)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()

    def work():
        s2.wait_stream(s1)
        with torch.cuda.stream(s2):
            for _ in range(4):
                big.mul_(1.0)
            v.copy_(src)
        with torch.cuda.stream(s1):
            q.copy_(src)
            mb.moa_attn_fwd(desc, q, q, q, O, L, stream=s1)
            s1.wait_stream(s2)
            mb.moa_attn_fwd(desc, q, q, v, O, L, stream=s1)

    torch.cuda.synchronize()
    with torch.cuda.stream(s1):
        work()
    s1.synchronize()
    if captured:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s1):
            work()
        run = g.replay
    else:
        def run():
            with torch.cuda.stream(s1):
                work()
    for _ in range(10):
        torch.cuda.synchronize()
        q.zero_(); v.zero_(); O.zero_()
        torch.cuda.synchronize()
        run()
        torch.cuda.synchronize()
        assert torch.equal(O, ref) and torch.equal(L, Lr)
