"""The stage-wise tests run with the stage tap open.  Its copies stand between launches that otherwise run beside each other, and f32 blocks keep a launch per
einsum with dbias in the first; what a program runs has the tap closed.  Both have to give the same bits."""
import pytest

from test_gpu_einsum import layout, mtf  # noqa: F401

pytestmark = pytest.mark.gpu

DIMS = {"x": ["t", "d"], "w": ["d", "f"], "v": ["f", "d"], "dy": ["t", "d"], "h": ["t", "f"], "dx": ["t", "d"], "dw": ["d", "f"], "dbias": ["f"], "dv": ["f", "d"]}


# bf16: several waves of pairs, sizes that no tile divides in slices, few tiles; f32: in pieces (whole tiles and ragged), on plain tiles, one launch a direction
@pytest.mark.parametrize("dtype,T,D,F,slices", [("bf16", 4096, 1024, 4096, 8), ("bf16", 1665, 776, 3080, 1), ("bf16", 128, 1024, 4096, 8), ("bf16", 96, 256, 512, 1),
                                                ("f32", 1024, 256, 1024, 4), ("f32", 520, 200, 904, 1), ("f32", 48, 64, 256, 1), ("f32", 8, 64, 256, 4)])
@pytest.mark.parametrize("bias", [True, False])
def test_feed_forward_backward(mtf, dtype, T, D, F, slices, bias):  # noqa: F811
    import torch
    g = torch.Generator(device="cuda").manual_seed(6)
    act = torch.bfloat16 if dtype == "bf16" else torch.float32
    t = {k: (torch.randn(*s, generator=g, device="cuda") * c).to(act) for k, s, c in
         (("x", (T, D), 1.0), ("w", (D, F), D ** -0.5), ("v", (F, D), F ** -0.5), ("dy", (T, D), 1.0), ("h", (T, F), 1.0))}
    t["h"].relu_()
    for k, s, dt in (("dx", (T, D), act), ("dw", (D, F), torch.float32), ("dbias", (F,), torch.float32), ("dv", (F, D), torch.float32)):
        t[k] = torch.empty(*s, dtype=dt, device="cuda")
    n = {k: mtf.named(v, DIMS[k]) for k, v in t.items()}
    if not bias:
        n["dbias"] = None
    lay = layout(mtf, [("p", slices)], [("f", "p")] if slices > 1 else [])
    ws = torch.empty(mtf.mtf_ffn_workspace_bytes(lay, n["x"], n["w"]), dtype=torch.uint8, device="cuda")
    buf = torch.empty(T * F * 4 + 4096, dtype=torch.uint8, device="cuda")
    outs = [k for k in ("dx", "dw", "dbias", "dv") if n[k] is not None]

    def run(tap):
        for k in outs:
            t[k].fill_(float("nan"))
        ws.fill_(0xFF)
        if tap:
            mtf.mtf_stage_tap_begin(buf)
        mtf.mtf_ffn_backward(lay, n["x"], n["w"], n["v"], n["h"], n["dy"], n["dx"], n["dw"], n["dbias"], n["dv"], ws)
        if tap:
            assert mtf.mtf_stage_tap_end() == 1
        mtf.mtf_device_status()
        return {k: t[k].clone() for k in outs}

    open_, closed = run(True), [run(False) for _ in range(3)]
    dhp = buf[mtf.mtf_stage_tap_entry(0)[1]:][:T * F * t["h"].element_size()].view(act).view(T, F).double()
    for k in outs:
        for c in closed:
            if k == "dbias" and dtype == "f32":      # summed by another launch: at most T roundings of 2^-24 of what was added up
                assert ((c[k].double() - dhp.sum(0)).abs() <= T * 2.0 ** -24 * dhp.abs().sum(0)).all()
            else:
                assert torch.equal(c[k], open_[k]), k
