"""The f32 feed-forward block and the attention block on its core by rows, captured into a graph, on a second stream, and from
two threads at once on a stream each (one layout, hence one plan cache): every output repeats the serial call's bits."""
import threading

import pytest

import seeded_inputs as si
from helpers import to_torch

pytestmark = pytest.mark.gpu


def _block(kind, seed, lay):
    """(step, outputs) of one block's forward and backward pass on tensors of its own."""
    import torch
    import paper_1811_02084_b200 as mtf
    act, N = ["batch", "length", "d_model"], mtf.named
    n, outs = {}, []

    def put(name, shape, dims, dtype, scale=1.0):
        n[name] = N(to_torch(si.normal(seed, name, shape, dtype, scale)), dims)

    def room(name, shape, dims, dtype):
        t = torch.full(shape, float("nan"), dtype=dtype, device="cuda")
        n[name] = N(t, dims)
        outs.append(t)

    if kind == "ffn f32":
        B, L, D, F, dt = 8, 8, 64, 256, torch.float32             # (one tile of tokens: its bias gradient has one order too)
        put("x", [B, L, D], act, "f32")
        put("dy", [B, L, D], act, "f32")
        put("w", [D, F], ["d_model", "d_ff"], "f32", D ** -0.5)
        put("v", [F, D], ["d_ff", "d_model"], "f32", F ** -0.5)
        put("bias", [F], ["d_ff"], "f32", 0.1)
        for name, shape, dims in (("h", (B, L, F), ["batch", "length", "d_ff"]), ("y", (B, L, D), act), ("dx", (B, L, D), act), ("dw", (D, F), ["d_model", "d_ff"]),
                                  ("dv", (F, D), ["d_ff", "d_model"]), ("dbias", (F,), ["d_ff"])):
            room(name, shape, dims, dt)
        ws = torch.empty(mtf.mtf_ffn_workspace_bytes(lay, n["x"], n["w"]), dtype=torch.uint8, device="cuda")

        def step():
            mtf.mtf_ffn_forward(lay, n["x"], n["w"], n["bias"], n["v"], n["h"], n["y"], ws)
            mtf.mtf_ffn_backward(lay, n["x"], n["w"], n["v"], n["h"], n["dy"], n["dx"], n["dw"], n["dbias"], n["dv"], ws)
        return step, outs
    B, L, D, H, K = 2, 456, 128, 4, 64
    bf, f32 = torch.bfloat16, torch.float32
    put("x", [B, L, D], act, "bf16")
    put("dy", [B, L, D], act, "bf16")
    for w, last in (("wq", "d_k"), ("wk", "d_k"), ("wv", "d_v")):
        put(w, [D, H, K], ["d_model", "heads", last], "bf16", D ** -0.5)
        room("d" + w, (D, H, K), ["d_model", "heads", last], f32)
    put("wo", [H, K, D], ["heads", "d_v", "d_model"], "bf16", (H * K) ** -0.5)
    room("dwo", (H, K, D), ["heads", "d_v", "d_model"], f32)
    for name, m, last in (("q", "length", "d_k"), ("kk", "memory_length", "d_k"), ("vv", "memory_length", "d_v"), ("o", "length", "d_v")):
        room(name, (B, L, H, K), ["batch", m, "heads", last], bf)
    room("weights", (B, H, L, L), ["batch", "heads", "length", "memory_length"], bf)
    room("y", (B, L, D), act, bf)
    room("dx", (B, L, D), act, bf)
    ws = torch.empty(mtf.mtf_attention_workspace_bytes(lay, n["x"], n["wq"], n["wv"]), dtype=torch.uint8, device="cuda")

    def step():
        mtf.mtf_attention_forward(lay, n["x"], n["wq"], n["wk"], n["wv"], n["wo"], True, None, n["q"], n["kk"], n["vv"], n["weights"], n["o"], n["y"], ws)
        mtf.mtf_attention_backward(lay, n["x"], n["wq"], n["wk"], n["wv"], n["wo"], n["q"], n["kk"], n["vv"], n["weights"], n["o"], n["dy"], None, n["dx"], n["dwq"],
                                   n["dwk"], n["dwv"], n["dwo"], ws, causal=True)
    return step, outs


@pytest.mark.parametrize("kind", ["ffn f32", "attention by rows"])
def test_graph_second_stream_and_two_threads(kind):
    import torch
    import paper_1811_02084_b200 as mtf
    lay = mtf.mtf_layout(mtf.mtf_mesh_create([("all", 1)]), [])
    blocks = [_block(kind, seed, lay) for seed in (31, 32)]
    for step, _ in blocks:
        step()
    mtf.mtf_device_status()
    want = [[t.clone() for t in outs] for _, outs in blocks]
    assert all(bool(torch.isfinite(t).all()) for w in want for t in w)

    def same(what):
        mtf.mtf_device_status()
        for w, (_, outs) in zip(want, blocks):
            for i, (a, b) in enumerate(zip(w, outs)):
                assert torch.equal(a, b), (what, i)
                b.zero_()
        torch.cuda.synchronize()

    same("eager")
    streams = [torch.cuda.Stream() for _ in blocks]
    for (step, _), s in zip(blocks, streams):
        with torch.cuda.stream(s):
            step()
    same("streams")
    errors = []

    def work(i):
        try:
            with torch.cuda.stream(streams[i]):
                for _ in range(20):
                    blocks[i][0]()
        except Exception as e:      # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    same("threads")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for step, _ in blocks:
            step()
    for rep in range(2):
        graph.replay()
        same(("graph", rep))
