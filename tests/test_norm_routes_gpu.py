"""RMSNorm on both sides of the lines between its register and its ring kernels (rows of 256..2048 elements; by n times d, another line
in the forward than in the backward) and of the line up to which the backward is one launch, with ragged numbers of rows and row lengths that
leave vectors over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import oracle
from paper_2609_33916_b200 import inputs as mi

TOL = 1e-2        # bf16 storage, fp32 arithmetic: the bound of the other RMSNorm tests


@pytest.mark.parametrize("n,d", [(4096, 256), (4097, 256), (511, 2048), (513, 2048), (1033, 1016), (127, 264), (32767, 256), (32801, 256),
                                 (8300, 1016), (768, 64), (769, 64), (1, 8), (33, 72), (700, 4104)])
def test_rmsnorm_routes(n, d):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    build.build()
    inp = mi.make_norm_inputs(n, d, seed=7 * n + d)
    x, g, dy = (torch.from_numpy(np.ascontiguousarray(inp[k])).view(torch.bfloat16).cuda() for k in ("x", "g", "dy"))
    y, dx, dg = (torch.full_like(t, float("nan")) for t in (x, x, g))
    r = torch.full((n,), float("nan"), dtype=torch.float32, device="cuda")
    desc = mb.make_rmsnorm_desc(n, d, 1e-5)
    ws = torch.full((mb.moa_rmsnorm_workspace_bytes(desc),), 0xFF, dtype=torch.uint8, device="cuda")
    mb.moa_rmsnorm_fwd(desc, x, g, y, r)
    mb.moa_rmsnorm_bwd(desc, x, g, r, dy, dx, dg, ws)
    f = {k: mi.to_f64(v, "bf16") for k, v in inp.items()}
    ref = oracle.rmsnorm_fwd_bwd(f["x"], f["g"], f["dy"], 1e-5)
    for k, t in (("y", y), ("dx", dx), ("dg", dg)):
        got = t.float().cpu().numpy().astype(np.float64)
        assert np.all(np.isfinite(got)) and mi.rel_err(got, ref[k]) <= TOL, (k, mi.rel_err(got, ref[k]))
    assert mi.rel_err(r.cpu().numpy().astype(np.float64), ref["r"]) <= 1e-5


@pytest.mark.parametrize("with_r", [True, False])
@pytest.mark.parametrize("with_add", [True, False])
@pytest.mark.parametrize("n,d", [(513, 2048), (4099, 264), (1033, 1016), (8193, 136), (1537, 2056), (800, 4104), (900, 8192), (300, 72)])
def test_rmsnorm_backward_forms(n, d, with_add, with_r):
    """With and without the added gradient and the stored r, in the ring kernel (first three), the register kernels and the one-launch form."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2609_33916_b200 import binding as mb
    from paper_2609_33916_b200 import build
    build.build()
    inp = mi.make_norm_inputs(n, d, seed=5 * n + d)
    x, g, dy = (torch.from_numpy(np.ascontiguousarray(inp[k])).view(torch.bfloat16).cuda() for k in ("x", "g", "dy"))
    add = torch.randn(x.shape, generator=torch.Generator(device="cuda").manual_seed(n), device="cuda").bfloat16() if with_add else None
    y, dx, dg = (torch.full_like(t, float("nan")) for t in (x, x, g))
    r = torch.full((n,), float("nan"), dtype=torch.float32, device="cuda")
    desc = mb.make_rmsnorm_desc(n, d, 1e-5)
    ws = torch.full((mb.moa_rmsnorm_workspace_bytes(desc),), 0xFF, dtype=torch.uint8, device="cuda")
    mb.moa_rmsnorm_fwd(desc, x, g, y, r)
    mb.moa_rmsnorm_bwd(desc, x, g, r if with_r else None, dy, dx, dg, ws, dx_add=add)
    f = {k: mi.to_f64(v, "bf16") for k, v in inp.items()}
    ref = oracle.rmsnorm_fwd_bwd(f["x"], f["g"], f["dy"], 1e-5)
    want = ref["dx"] + (add.double().cpu().numpy() if with_add else 0.0)
    for got, r_ in ((dx, want), (dg, ref["dg"])):
        got = got.float().cpu().numpy().astype(np.float64)
        assert np.all(np.isfinite(got)) and mi.rel_err(got, r_) <= TOL


@pytest.mark.parametrize("n,d", [(2032, 1032), (2033, 1032), (1638, 1280), (1639, 1280), (2100, 1288)])
def test_rmsnorm_rows_above_1024(n, d):
    """Both sides of the forward's other line, for rows of 1032..1280 elements, and the first rows past them."""
    test_rmsnorm_routes(n, d)
