"""The attention core by rows (heads of 64 and 128 columns, rows of any length that is a multiple of 8) against plain fp64
arithmetic on the inputs each launch read: one and several key blocks, logits kept (up to 384 keys) and computed twice,
causal and not, lengths inside, on and just past a block, several pairs per SM."""
import pytest

import seeded_inputs as si
from helpers import TOL, Guarded, parity_error, from_torch, to_torch

pytestmark = pytest.mark.gpu

CASES = [(1, 1, 8, 64), (3, 2, 40, 64), (2, 3, 136, 64), (2, 2, 200, 128), (1, 2, 384, 128), (1, 2, 392, 64), (2, 1, 640, 128), (1, 2, 1000, 64), (40, 4, 72, 128)]


@pytest.mark.parametrize("B,H,L,D", CASES)
@pytest.mark.parametrize("causal", [False, True])
@pytest.mark.parametrize("tap", [False, True])
def test_forward_and_backward(B, H, L, D, causal, tap):
    import torch
    import paper_1811_02084_b200 as mtf
    M = 64                                                       # model width
    lay = mtf.mtf_layout(mtf.mtf_mesh_create([("all", 1)]), [])
    g = Guarded()
    n, t = {}, {}

    def put(name, s, dims):
        t[name], n[name] = to_torch(s), None
        n[name] = mtf.named(t[name], dims)

    def room(name, shape, dims, dtype="bf16"):
        t[name] = g.empty(shape, dtype)
        n[name] = mtf.named(t[name], dims)

    words, heads = ["batch", "length", "d_model"], {"q": ["batch", "length", "heads", "d_k"], "kk": ["batch", "memory_length", "heads", "d_k"],
                                                    "vv": ["batch", "memory_length", "heads", "d_v"], "o": ["batch", "length", "heads", "d_v"]}
    put("x", si.normal(1, "x", [B, L, M], "bf16"), words)
    put("dy", si.normal(1, "dy", [B, L, M], "bf16"), words)
    for w, last in (("wq", "d_k"), ("wk", "d_k"), ("wv", "d_v")):
        put(w, si.normal(1, w, [M, H, D], "bf16", 2 * M ** -0.5), ["d_model", "heads", last])
        room("d" + w, [M, H, D], ["d_model", "heads", last], "f32")
    put("wo", si.normal(1, "wo", [H, D, M], "bf16", (H * D) ** -0.5), ["heads", "d_v", "d_model"])
    room("dwo", [H, D, M], ["heads", "d_v", "d_model"], "f32")
    for name, dims in heads.items():
        room(name, [B, L, H, D], dims)
    room("weights", [B, H, L, L], ["batch", "heads", "length", "memory_length"])
    room("y", [B, L, M], words)
    room("dx", [B, L, M], words)
    ws = torch.empty(mtf.mtf_attention_workspace_bytes(lay, n["x"], n["wq"], n["wv"]), dtype=torch.uint8, device="cuda")
    ws.fill_(0xFF)                                               # (NaN in both types: what is read before it is written shows)
    before = mtf.mtf_launch_count()
    mtf.mtf_attention_forward(lay, n["x"], n["wq"], n["wk"], n["wv"], n["wo"], causal, None, n["q"], n["kk"], n["vv"], n["weights"], n["o"], n["y"], ws)
    assert mtf.mtf_launch_count() - before == 3                  # projections, core, output projection
    buf = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    args = [lay] + [n[k] for k in ("x", "wq", "wk", "wv", "wo", "q", "kk", "vv", "weights", "o", "dy")] + [None] + [n[k] for k in ("dx", "dwq", "dwk", "dwv", "dwo")]
    ws.fill_(0xFF)
    mtf.mtf_attention_backward(*args, ws, causal=causal)
    assert all(bool(torch.isfinite(t[k]).all()) for k in ("dx", "dwq", "dwk", "dwv", "dwo"))
    first = {k: t[k].clone() for k in ("dx", "dwq", "dwk", "dwv", "dwo")}
    if tap:
        mtf.mtf_stage_tap_begin(buf)
        mtf.mtf_attention_backward(*args, ws, causal=causal)
        stages = {}
        for i in range(mtf.mtf_stage_tap_end()):
            name, off, size = mtf.mtf_stage_tap_entry(i)
            stages[name] = buf[off:off + size]
        for k, v in first.items():
            assert torch.equal(v, t[k]), k                       # the tap changes nothing
    mtf.mtf_device_status()
    g.check()
    q, kk, vv, P = (t[k].double() for k in ("q", "kk", "vv", "weights"))
    z = torch.einsum("blhk,bmhk->bhlm", q, kk) * D ** -0.5
    if causal:
        z.masked_fill_(torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1), float("-inf"))
    assert parity_error(from_torch(t["weights"]), torch.softmax(z, -1).cpu().numpy()) <= TOL["bf16"]
    assert parity_error(from_torch(t["o"]), torch.einsum("bhlm,bmhv->blhv", P, vv).cpu().numpy()) <= TOL["bf16"]
    if not tap:
        return
    got = {k: stages[k].view(torch.bfloat16) for k in ("do", "dlogits", "dq", "dkk", "dvv")}
    do, ds = got["do"].double().view(B, L, H, D), got["dlogits"].double().view(B, H, L, L)
    dP = torch.einsum("blhv,bmhv->bhlm", do, vv)
    want = {"dlogits": P * (dP - (dP * P).sum(-1, keepdim=True)), "dq": torch.einsum("bhlm,bmhk->blhk", ds, kk) * D ** -0.5,
            "dkk": torch.einsum("bhlm,blhk->bmhk", ds, q) * D ** -0.5, "dvv": torch.einsum("bhlm,blhv->bmhv", P, do)}
    for k, ref in want.items():
        assert parity_error(from_torch(got[k].view(ref.shape)), ref.cpu().numpy()) <= TOL["bf16"], k


@pytest.mark.parametrize("L,D,bad", [(200, 64, (0, 32)), (200, 128, (64, 96)), (200, 64, (128, 200)), (640, 64, (0, 128)), (640, 64, (256, 384)), (1000, 128, (7, 8))])
@pytest.mark.parametrize("causal", [False, True])
def test_rows_with_a_nan_are_nan(L, D, bad, causal):
    """Positions whose q, kk and vv are NaN (whole groups of the columns a warp walks, and a single one): every row that sees
    one has NaN weights, as softmax gives; rows that see none, and weights right of the diagonal, are untouched."""
    import torch
    import paper_1811_02084_b200 as mtf
    lay = mtf.mtf_layout(mtf.mtf_mesh_create([("all", 1)]), [])
    B, H, M, bf = 1, 2, 64, torch.bfloat16
    torch.manual_seed(2)
    x = torch.randn(B, L, M, device="cuda").to(bf)
    x[:, bad[0]:bad[1]] = float("nan")
    words = ["batch", "length", "d_model"]
    w = [mtf.named((torch.randn(M, H, D, device="cuda") * M ** -0.5).to(bf), ["d_model", "heads", k]) for k in ("d_k", "d_k", "d_v")]
    wo = mtf.named(torch.randn(H, D, M, device="cuda").to(bf), ["heads", "d_v", "d_model"])
    q, kk, vv, o = (torch.empty(B, L, H, D, dtype=bf, device="cuda") for _ in range(4))
    P, y = torch.empty(B, H, L, L, dtype=bf, device="cuda"), torch.empty(B, L, M, dtype=bf, device="cuda")
    n = [mtf.named(t, ["batch", m, "heads", k]) for t, m, k in ((q, "length", "d_k"), (kk, "memory_length", "d_k"), (vv, "memory_length", "d_v"))]
    ws = torch.empty(mtf.mtf_attention_workspace_bytes(lay, mtf.named(x, words), w[0], w[2]), dtype=torch.uint8, device="cuda")
    before = mtf.mtf_launch_count()
    mtf.mtf_attention_forward(lay, mtf.named(x, words), *w, wo, causal, None, *n, mtf.named(P, ["batch", "heads", "length", "memory_length"]),
                              mtf.named(o, ["batch", "length", "heads", "d_v"]), mtf.named(y, words), ws)
    assert mtf.mtf_launch_count() - before == 3
    mtf.mtf_device_status()
    z = torch.einsum("blhk,bmhk->bhlm", q.double(), kk.double()) * D ** -0.5
    right = torch.ones(L, L, dtype=torch.bool, device="cuda").triu(1) if causal else torch.zeros(L, L, dtype=torch.bool, device="cuda")
    ref = torch.softmax(z.masked_fill(right, float("-inf")), -1).masked_fill(right, 0.0)
    assert torch.equal(P.isnan(), ref.isnan())
    assert parity_error(from_torch(P.nan_to_num(0.0)), ref.nan_to_num(0.0).cpu().numpy()) <= TOL["bf16"]
