"""Outputs laid over inputs that no later kernel of the call reads: small calls, whose kernels may run side by side, give the bits that separate
buffers give, whichever launches they take."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    torch = pytest.importorskip("torch")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    build.build()
    return torch, mb


def _mlp(torch, n, d, dff):
    gen = torch.Generator(device="cuda").manual_seed(n)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    t = {"x": R(n, d), "W1": R(dff, d) * d ** -0.5, "W3": R(dff, d) * d ** -0.5, "W2": R(d, dff) * dff ** -0.5, "a": R(n, dff), "u": R(n, dff),
         "h": R(n, dff), "dy": R(n, d)}
    out = {"dx": (n, d), "dW1": (dff, d), "dW3": (dff, d), "dW2": (d, dff)}
    return t, out


def _bwd(torch, mb, n, d, dff, t, out):
    desc = mb.make_mlp_desc(n, d, dff)
    ws = torch.empty(mb.moa_gated_mlp_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
    before = mb.moa_launch_count()
    mb.moa_gated_mlp_bwd(desc, *(t[k] for k in ("x", "W1", "W3", "W2", "a", "u", "h", "dy")), *(out[k] for k in ("dx", "dW1", "dW3", "dW2")), ws)
    launches = mb.moa_launch_count() - before
    assert mb.moa_last_device_status() == mb.MOA_OK
    return {k: v.clone() for k, v in out.items()}, launches


# (output, input it lies over, elements it is shifted by): behind the launch that reads the input when the products go one after the other
@pytest.mark.parametrize("over,under,shift", [("dx", "dy", 0), ("dx", "x", 0), ("dx", "h", 0), ("dx", "x", 64), ("dx", "dy", 320),
                                              ("dW1", "dy", 0), ("dW3", "h", 64), ("dW1", "h", 0)])
@pytest.mark.parametrize("n,d,dff", [(300, 64, 256), (512, 128, 320), (40, 64, 40)])
def test_gated_mlp_backward(rt, n, d, dff, over, under, shift):
    torch, mb = rt
    t, shapes = _mlp(torch, n, d, dff)
    E = lambda k: torch.empty(shapes[k], dtype=torch.bfloat16, device="cuda")      # noqa: E731
    ref, grouped = _bwd(torch, mb, n, d, dff, t, {k: E(k) for k in shapes})
    assert grouped == 2
    count = shapes[over][0] * shapes[over][1]
    pool = torch.empty(max(t[under].numel(), count) + shift, dtype=torch.bfloat16, device="cuda")
    # the output begins `shift` elements behind the input
    pool[:t[under].numel()] = t[under].flatten()
    tt = dict(t, **{under: pool[:t[under].numel()].view(t[under].shape)})
    out = {k: E(k) for k in shapes if k != over}
    out[over] = pool[shift:shift + count].view(shapes[over])
    got, launches = _bwd(torch, mb, n, d, dff, tt, out)
    assert launches == 4
    for k in shapes:
        assert torch.equal(got[k], ref[k]), k


def test_block_weight_gradient_over_the_weight(rt):
    """dWqkv over Wqkv, which dh1 reads first."""
    torch, mb = rt
    from paper_2609_33916_b200.block import TransformerBlock
    B, n, H, d, dff = 1, 200, 1, 64, 128
    gen = torch.Generator(device="cuda").manual_seed(5)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    dm = H * d
    w = {k: R(dm, dm) * dm ** -0.5 for k in ("Wq", "Wk", "Wv", "Wo")}
    w.update(W1=R(dff, dm) * dm ** -0.5, W3=R(dff, dm) * dm ** -0.5, W2=R(dm, dff) * dff ** -0.5, g1=1 + 0.25 * R(dm), g2=1 + 0.25 * R(dm))
    x, dy = R(B * n, dm), R(B * n, dm)
    res = []
    for over in (False, True):
        blk = TransformerBlock(torch, B, n, H, d, dff, True)
        wp = blk.prepare_weights(w)
        blk.forward(x, wp)
        if over:
            blk.gqkv = wp["Wqkv"]
        before = mb.moa_launch_count()
        dx, _ = blk.backward(x, wp, dy)
        res.append((dx.double(), blk.gqkv.double(), mb.moa_launch_count() - before))
    assert res[1][2] == res[0][2] + 1
    for a, b in zip(res[0][:2], res[1][:2]):      # (dQ's atomic sums in another order, and their bf16 roundings down the chain)
        assert (a - b).abs().max().item() <= 1.6e-2 * a.abs().max().item()


# register kernel with one and with several CTAs; dx over x or dy row for row; dg over what the other rows' CTAs still read
@pytest.mark.parametrize("over,under", [("dx", "x"), ("dx", "dy"), ("dx", "dx_add"), ("dg", "g"), ("dg", "x"), ("dg", "dy"), ("dg", "dx_add"), ("dg", "r")])
@pytest.mark.parametrize("n,d", [(700, 64), (512, 1024), (64, 72), (1, 256)])
def test_rmsnorm_backward(rt, n, d, over, under):
    torch, mb = rt
    gen = torch.Generator(device="cuda").manual_seed(n + d)
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    t = {"x": R(n, d), "g": 1 + 0.25 * R(d), "dy": R(n, d), "dx_add": R(n, d), "r": torch.empty(n, dtype=torch.float32, device="cuda")}
    desc = mb.make_rmsnorm_desc(n, d, 1e-5)
    mb.moa_rmsnorm_fwd(desc, t["x"], t["g"], torch.empty_like(t["x"]), t["r"])
    if t[under].nbytes < 2 * d:
        pytest.skip("the output does not fit into this input")

    def run(reused):
        a = {k: v.clone() for k, v in t.items()}
        out = {"dx": torch.empty_like(a["x"]), "dg": torch.empty_like(a["g"])}
        if reused:
            like = out[over]
            out[over] = a[under].view(torch.bfloat16).flatten()[:like.numel()].view(like.shape)
        ws = torch.empty(mb.moa_rmsnorm_workspace_bytes(desc), dtype=torch.uint8, device="cuda")
        before = mb.moa_launch_count()
        mb.moa_rmsnorm_bwd(desc, a["x"], a["g"], a["r"], a["dy"], out["dx"], out["dg"], ws, dx_add=a["dx_add"])
        return out["dx"].double(), out["dg"].double(), mb.moa_launch_count() - before

    ref, got = run(False), run(True)
    assert ref[2] == 1 and got[2] == (1 if under == "dx_add" and over == "dx" else 2)
    # dx does not depend on the route; dg's sums are taken in another order: fp32 sums of n terms, then one rounding to bf16 (2^-8 of an element)
    assert torch.equal(ref[0], got[0])
    assert (ref[1] - got[1]).abs().max().item() <= 2 ** -7 * ref[1].abs().max().item()
