"""Blocks whose outputs lie over operands that no later product reads: the products that share memory run one behind another, so every output has the bits that
it has on buffers of its own."""
import pytest

from test_gpu_einsum import layout, mtf  # noqa: F401

pytestmark = pytest.mark.gpu

DIMS = {"x": ["t", "d"], "w": ["d", "f"], "v": ["f", "e"], "dy": ["t", "e"], "h": ["t", "f"], "dx": ["t", "d"], "dw": ["d", "f"], "dbias": ["f"], "dv": ["f", "e"]}


def ffn_operands(dtype, T, D, F):
    import torch
    g = torch.Generator(device="cuda").manual_seed(3)
    t = {k: (torch.randn(*s, generator=g, device="cuda") * c).to(dtype) for k, s, c in
         (("x", (T, D), 1.0), ("w", (D, F), D ** -0.5), ("v", (F, D), F ** -0.5), ("dy", (T, D), 1.0), ("h", (T, F), 1.0))}
    t["h"].relu_()
    return t


def ffn_backward(mtf, t, dtype, T, D, F, bias, over):  # noqa: F811
    """over: output -> operand (or output) whose memory it takes."""
    import torch
    f32 = torch.float32
    out = {"dx": ((T, D), dtype), "dw": ((D, F), f32), "dbias": ((F,), f32), "dv": ((F, D), f32)}
    for k, (shape, dt) in out.items():
        n = torch.Size(shape).numel() * (2 if dt == torch.bfloat16 else 4)
        if k in over:                     # room for both: the operand moves to the head of a buffer of the larger size
            src = t[over[k]]
            buf = torch.empty(max(n, src.numel() * src.element_size()), dtype=torch.uint8, device="cuda")
            moved = buf[:src.numel() * src.element_size()].view(src.dtype).view(src.shape)
            moved.copy_(src)
            t[over[k]] = moved
            t[k] = buf[:n].view(dt).view(shape)
        else:
            t[k] = torch.full(shape, float("nan"), dtype=dt, device="cuda")
    if not bias:
        t["dbias"] = None
    n = {k: None if v is None else mtf.named(v, DIMS[k]) for k, v in t.items()}
    lay = layout(mtf, [("all", 1)], [])
    ws = torch.empty(mtf.mtf_ffn_workspace_bytes(lay, n["x"], n["w"]), dtype=torch.uint8, device="cuda")
    mtf.mtf_ffn_backward(lay, n["x"], n["w"], n["v"], n["h"], n["dy"], n["dx"], n["dw"], n["dbias"], n["dv"], ws)
    mtf.mtf_device_status()
    return {k: t[k].clone() for k in out if t[k] is not None}


# bf16: products of several waves on pairs, of few tiles on the 128-row kernel; f32: products in pieces, and the size that is one launch where nothing overlaps
@pytest.mark.parametrize("dtype,T,D,F", [("bf16", 2048, 1024, 4096), ("bf16", 160, 512, 2048), ("f32", 1024, 256, 1024), ("f32", 8, 64, 256)])
@pytest.mark.parametrize("over", [{"dv": "v"}, {"dx": "x"}, {"dv": "v", "dx": "x"}, {"dx": "dy"}, {"dx": "h", "dv": "v"}])
@pytest.mark.parametrize("bias", [True, False])
def test_feed_forward_backward(mtf, dtype, T, D, F, over, bias):  # noqa: F811
    import torch
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    first = ffn_operands(dt, T, D, F)
    want = ffn_backward(mtf, dict(first), dt, T, D, F, bias, {})
    for _ in range(3):
        got = ffn_backward(mtf, dict(first), dt, T, D, F, bias, over)
        for k, v in want.items():
            if dtype == "bf16" or k != "dbias":
                assert torch.equal(got[k], v) if (dtype, T) != ("f32", 8) else (got[k].double() - v.double()).norm() <= 1e-6 * v.double().norm(), k
            else:                         # added to memory in an order that varies where launches stand alone
                assert (got[k].double() - v.double()).norm() <= 1e-6 * v.double().norm(), k


def test_a_later_product_reads_what_an_earlier_one_wrote(mtf):  # noqa: F811
    import torch
    T, D, F = 1024, 256, 1024
    t = ffn_operands(torch.float32, T, D, F)
    got = ffn_backward(mtf, t, torch.float32, T, D, F, True, {"dw": "w"})       # launch by launch dx = dhp . dw^T
    dhp = (t["dy"].double() @ t["v"].double().t()) * (t["h"] > 0)
    ref = dhp @ got["dw"].double().t()
    assert (got["dx"].double() - ref).norm() <= 1e-6 * ref.norm()


# rows of 512 (one-launch core), of 200 (core by rows) and of 136 with heads of 32 (launch by launch)
@pytest.mark.parametrize("B,L,M,H,K", [(8, 512, 1024, 16, 64), (3, 200, 512, 8, 64), (2, 136, 256, 4, 32)])
@pytest.mark.parametrize("over", [{"dx": "x"}, {"dwk": "kk"}, {"dx": "x", "dwv": "weights"}, {"dx": "dy"}])
def test_attention_backward(mtf, B, L, M, H, K, over):  # noqa: F811
    import torch
    g = torch.Generator(device="cuda").manual_seed(4)
    words, f32 = ["batch", "length", "d_model"], torch.float32
    shapes = {"x": ((B, L, M), words), "dy": ((B, L, M), words), "y": ((B, L, M), words), "wo": ((H, K, M), ["heads", "d_v", "d_model"]),
              "weights": ((B, H, L, L), ["batch", "heads", "length", "memory_length"])}
    shapes |= {w: ((M, H, K), ["d_model", "heads", "d_v" if w == "wv" else "d_k"]) for w in ("wq", "wk", "wv")}
    shapes |= {a: ((B, L, H, K), ["batch", "length" if a in ("q", "o") else "memory_length", "heads", "d_v" if a in ("vv", "o") else "d_k"]) for a in ("q", "kk", "vv", "o")}
    first = {k: (torch.randn(*s, generator=g, device="cuda") * (M ** -0.5 if k[0] == "w" and k != "weights" else 1.0)).bfloat16() for k, (s, _) in shapes.items()}
    lay = layout(mtf, [("all", 1)], [])
    named = {k: mtf.named(first[k], shapes[k][1]) for k in shapes}
    ws = torch.empty(mtf.mtf_attention_workspace_bytes(lay, named["x"], named["wq"], named["wv"]), dtype=torch.uint8, device="cuda")
    mtf.mtf_attention_forward(lay, *[named[k] for k in ("x", "wq", "wk", "wv", "wo")], False, None, *[named[k] for k in ("q", "kk", "vv", "weights", "o", "y")], ws)

    def backward(over):
        t = dict(first)
        out = {"dx": ("x", torch.bfloat16), "dwq": ("wq", f32), "dwk": ("wk", f32), "dwv": ("wv", f32), "dwo": ("wo", f32)}
        for k, (like, dt) in out.items():
            size = first[like].numel() * (2 if dt == torch.bfloat16 else 4)
            if k in over:
                src = first[over[k]]
                buf = torch.empty(max(size, src.numel() * 2), dtype=torch.uint8, device="cuda")
                t[over[k]] = buf[:src.numel() * 2].view(torch.bfloat16).view(src.shape)
                t[over[k]].copy_(src)
                t[k] = buf[:size].view(dt).view(first[like].shape)
            else:
                t[k] = torch.full(first[like].shape, float("nan"), dtype=dt, device="cuda")
        n = {k: mtf.named(v, shapes[out[k][0] if k in out else k][1]) for k, v in t.items()}
        mtf.mtf_attention_backward(lay, *[n[k] for k in ("x", "wq", "wk", "wv", "wo", "q", "kk", "vv", "weights", "o", "dy")], None,
                                   *[n[k] for k in ("dx", "dwq", "dwk", "dwv", "dwo")], ws)
        mtf.mtf_device_status()
        return {k: t[k].clone() for k in out}

    want = backward({})
    for _ in range(3):
        got = backward(over)
        assert all(torch.equal(got[k], want[k]) for k in want)
