"""Calls whose kernels start while their predecessors drain: chains of calls on reused buffers, behind a join of two
streams, under capture, give what the same calls give with a synchronisation after each.  Decode on every route (clusters, segments merged through
memory, whose kernel streams the cache before its own wait, the grouped kernel and its merge) behind a kernel that has just written its cache
and query; forward and backward that add into an accumulator which the kernel in front clears."""
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


# clusters | segments through memory behind the clearing kernel, single heads and the ring | grouped: a cluster, all SMs and a merge | the 128-row route
@pytest.mark.parametrize("dtype,B,H,Hkv,n,d", [("bf16", 1, 16, 16, 1000, 64), ("bf16", 1, 8, 8, 30000, 64), ("f32", 1, 8, 8, 12000, 64),
                                               ("f32", 1, 32, 8, 6000, 64), ("bf16", 1, 8, 1, 3000, 64), ("bf16", 1, 8, 1, 20000, 64),
                                               ("bf16", 1, 32, 1, 4000, 128)])
def test_decode_behind_a_cache_update(rt, dtype, B, H, Hkv, n, d):
    """Steps of a generation on one stream, one cache and one workspace: new keys and values are written over the whole cache, then the call."""
    torch, mb = rt
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(n)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").to(t)      # noqa: E731
    steps = 6
    caches, queries = [(R(B, Hkv, n, d), R(B, Hkv, n, d)) for _ in range(2)], [R(B, H, d) for _ in range(steps)]
    K, V, q = (torch.empty_like(x) for x in (caches[0][0], caches[0][1], queries[0]))
    desc = mb.make_decode_desc(B, H, n, d, d ** -0.5, mb.MOA_BF16 if dtype == "bf16" else mb.MOA_F32, H_kv=0 if H == Hkv else Hkv)
    ws = torch.empty(max(16, mb.moa_decode_workspace_bytes(desc)), dtype=torch.uint8, device="cuda")

    def run(between):
        out = []
        for i in range(steps):
            K.copy_(caches[i % 2][0]); V.copy_(caches[i % 2][1]); q.copy_(queries[i])
            between()
            o, lse = torch.empty_like(q), torch.empty((B, H), dtype=torch.float32, device="cuda")
            mb.moa_decode_attn(desc, q, K, V, o, lse, ws); between()
            mb.moa_decode_attn(desc, o, K, V, q, lse, ws); between()      # its query is the output of the call in front
            out += [o, q.clone(), lse]
        return out

    ref = run(torch.cuda.synchronize)
    for _ in range(10):
        got = run(lambda: None)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(got, ref))


# bf16: jobs of their own, shared key tiles, 64 columns, the one-pass and the two-pass wide backward, a long walk (an ordinary launch) | fp32 alone, in
# clusters, and where the forward is an ordinary launch
@pytest.mark.parametrize("dtype,B,H,Hkv,n,d", [("bf16", 2, 16, 16, 520, 128), ("bf16", 1, 8, 1, 900, 128), ("bf16", 2, 16, 16, 700, 64), ("bf16", 1, 4, 2, 500, 192),
                                               ("bf16", 1, 4, 4, 500, 256), ("bf16", 1, 16, 2, 900, 128), ("f32", 1, 1, 1, 128, 64), ("f32", 1, 2, 2, 583, 64),
                                               ("f32", 2, 16, 16, 300, 64)])
@pytest.mark.parametrize("fused", [True, False])
def test_accumulators_cleared_by_the_kernel_in_front(rt, dtype, B, H, Hkv, n, d, fused):
    """Calls in the default dq_mode, each on the outputs of the one before, one workspace and one set of outputs.  Everything but dQ has one writer
    and one order; dQ's is free: fp32 sums in another order, so within their rounding (bf16: one rounding of the result)."""
    torch, mb = rt
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(n + d)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").to(t)      # noqa: E731
    desc = mb.make_desc(B, H, n, d, True, d ** -0.5, mb.MOA_BF16 if dtype == "bf16" else mb.MOA_F32, H_kv=0 if H == Hkv else Hkv)
    ws = torch.empty(max(16, mb.moa_attn_workspace_bytes(desc, mb.MOA_OP_FUSED)), dtype=torch.uint8, device="cuda")
    Q0, K0, V0, dO0 = R(B, H, n, d), R(B, Hkv, n, d), R(B, Hkv, n, d), R(B, H, n, d)

    def run(between):
        Q, K, V, dO = Q0.clone(), K0.clone(), V0.clone(), dO0.clone()
        O, dQ, dK, dV = (torch.empty_like(x) for x in (Q, Q, K, V))
        L = torch.empty((B, H, n), dtype=torch.float32, device="cuda")
        out = []
        for _ in range(3):
            if fused:
                mb.moa_attn_fused_fwd_bwd(desc, Q, K, V, dO, O, L, dQ, dK, dV, ws); between()
            else:
                mb.moa_attn_fwd(desc, Q, K, V, O, L); between()
                mb.moa_attn_bwd(desc, Q, K, V, O, L, dO, dQ, dK, dV, ws); between()
            out.append([x.clone() for x in (O, L, dK, dV, dQ)])
            V.copy_(dK); K.copy_(dV); dO.copy_(O)      # (nothing of the free order goes on)
            between()
        return out

    ref = run(torch.cuda.synchronize)
    for _ in range(6):
        got = run(lambda: None)
        torch.cuda.synchronize()
        for a, b in zip(got, ref):
            assert all(torch.equal(x, y) for x, y in zip(a[:4], b[:4]))
            assert (a[4].double() - b[4].double()).abs().max().item() <= (2 ** -8 if dtype == "bf16" else 1e-5) * b[4].double().abs().max().item()
