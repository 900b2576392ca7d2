"""A block whose descriptors were changed after it was built (its attention's dq_mode or scale, its norms' eps) runs with the changed ones."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("field", ["dq_mode", "scale", "eps"])
def test_changed_descriptors(field):
    torch = pytest.importorskip("torch")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    from paper_2609_33916_b200.block import TransformerBlock
    build.build()
    B, n, H, d, dff = 2, 300, 2, 64, 136
    gen = torch.Generator(device="cuda").manual_seed(n)
    dm = H * d
    R = lambda *s: torch.randn(s, generator=gen, device="cuda").bfloat16()      # noqa: E731
    w = {k: R(dm, dm) * dm ** -0.5 for k in ("Wq", "Wk", "Wv", "Wo")}
    w.update(W1=R(dff, dm) * dm ** -0.5, W3=R(dff, dm) * dm ** -0.5, W2=R(dm, dff) * dff ** -0.5, g1=1 + 0.25 * R(dm), g2=1 + 0.25 * R(dm))
    x, dy = R(B * n, dm), R(B * n, dm)
    out = {}
    for packed in (True, False):
        blk = TransformerBlock(torch, B, n, H, d, dff, True, packed_qkv=packed)
        wp = blk.prepare_weights(w)
        plain = blk.forward(x, wp).clone()
        if field == "dq_mode":
            blk.ad.dq_mode = mb.MOA_DQ_SEPARATE_PASS
        elif field == "scale":
            blk.ad.scale *= 0.5
        else:
            blk.nd.eps = 0.5
        y = blk.forward(x, wp).clone()
        assert torch.equal(y, plain) == (field == "dq_mode")
        runs = []
        for _ in range(3):
            dx, g = blk.backward(x, wp, dy)
            runs.append([dx.clone()] + [t.clone() for t in (blk.dq, blk.dk, blk.dv)] + [g[k].clone() for k in sorted(g)])
        if field == "dq_mode":      # no atomics: the same bits every time
            assert all(torch.equal(a, b) for r in runs[1:] for a, b in zip(r, runs[0]))
            # dQ of the mode that was asked for, from the block's own tensors
            dq, dk, dv = (torch.empty_like(t) for t in (blk.dqkv,) * 3)
            if packed:
                third = lambda t: t.view(B, n, 3, H, d)[:, :, 0]      # noqa: E731
                mb.moa_attn_bwd(blk.ad, blk.q, blk.k, blk.v, blk.o, blk.L, blk.do, third(dq), third(dk), third(dv), blk.aws)
                assert torch.equal(third(dq), blk.dq)
        out[packed] = [y] + runs[0]
        assert mb.moa_last_device_status() == mb.MOA_OK
    assert torch.equal(out[True][0], out[False][0])
    for a, b in zip(out[True][1:], out[False][1:]):      # (dh1 is one sum of three there: bf16 results)
        a, b = a.double().reshape(-1), b.double().reshape(-1)
        assert (a - b).abs().max().item() <= 1.6e-2 * b.abs().max().item()
