"""The work that a user of this library has it do, as timed cases: the feed-forward block, the attention block, the decoder
layer and the vocabulary step, each through its entry points in the Python binding, on tensors that the caller keeps."""
import torch

import paper_1811_02084_b200 as mtf

MEMORY = "memory_length"
GRADS = {"wq": "dwq", "wk": "dwk", "wv": "dwv", "wo": "dwo", "ln1_gamma": "dln1_gamma", "ln1_beta": "dln1_beta", "w": "dw", "bias": "dbias", "v": "dv",
         "ln2_gamma": "dln2_gamma", "ln2_beta": "dln2_beta"}


def ffn(name, dtype, batch, length, d_model, d_ff, mesh, rules, backward=True):
    c = {"kind": "ffn", "dtype": dtype, "batch": batch, "length": length, "d_model": d_model, "d_ff": d_ff, "mesh": mesh, "rules": rules, "backward": backward}
    return {"name": name, **c} if name else c


def attention(name, batch, length, d_model, heads, d_k, causal, mesh, rules, backward=True):
    c = {"kind": "attention", "batch": batch, "length": length, "d_model": d_model, "heads": heads, "d_k": d_k, "causal": causal, "mesh": mesh, "rules": rules,
         "backward": backward}
    return {"name": name, **c} if name else c


def decoder(name, batch, length, d_model, heads, d_k, d_ff, mesh, rules, backward=True):
    c = {"kind": "decoder", "batch": batch, "length": length, "d_model": d_model, "heads": heads, "d_k": d_k, "d_ff": d_ff, "causal": True, "mesh": mesh,
         "rules": rules, "backward": backward}
    return {"name": name, **c} if name else c


def vocab(name, batch, length, d_model, words, mesh, rules):
    c = {"kind": "vocab", "batch": batch, "length": length, "d_model": d_model, "vocab": words, "mesh": mesh, "rules": rules}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the example of the method at toy size in 32 bits, on a 2 x 2 mesh: what a first program or a unit test runs; all latency
        ffn("ffn f32 toy", "f32", 1, 8, 64, 256, "2x2", "batch:0,d_ff:1") | {"batch": 8, "length": 1},
        # the same block in 32 bits at a size where the arithmetic counts: checking a layout's numbers before the bf16 run
        ffn("ffn f32", "f32", 8, 128, 256, 1024, "2x2", "batch:0,d_ff:1"),
        # one short sequence through a full-width block, as in fine-tuning or a per-rank slice of a small batch: few output tiles
        ffn("ffn few tokens", "bf16", 1, 128, 1024, 4096, "8", "d_ff:0"),
        # sizes that no tile divides, batch split
        ffn("ffn ragged", "bf16", 5, 333, 776, 3080, "5", "batch:0"),
        # the feed-forward block that the benchmark times: 32 sequences of 256 tokens, hidden units over 8 processors
        ffn("ffn", "bf16", 32, 256, 1024, 8192, "8", "d_ff:0"),
        # the widest model of the paper's tables: 65536 hidden units over 16 processors
        ffn("ffn wide", "bf16", 32, 256, 1024, 65536, "16", "d_ff:0"),
        # the attention block that the benchmark times: rows of 512, 16 heads of 64, batch and heads over a 4 x 4 mesh
        attention("attention", 16, 512, 1024, 16, 64, False, "4x4", "batch:0,heads:1"),
        # heads of 128 as in the paper's translation models, causal rows longer than a tile
        attention("attention heads of 128", 4, 1024, 1024, 8, 128, True, "2x2", "batch:0,heads:1"),
        # a few short sequences whose length no tile divides
        attention("attention ragged", 3, 200, 512, 8, 64, True, "1", ""),
        # the full decoder layer that the benchmark times: 64 sequences of 256 tokens, width 2048, batch and d_ff / heads over a 4 x 8 mesh
        decoder("decoder layer", 64, 256, 2048, 32, 64, 8192, "4x8", "batch:0,heads:1,d_ff:1"),
        # evaluation: the forward pass of one layer over two sequences, nothing split
        decoder("decoder forward", 2, 256, 1024, 16, 64, 4096, "1", "", backward=False),
        # both ends of the model over 32768 words: embedding, logits and loss, their gradients, and the update of both tables
        vocab("vocab step", 32, 256, 1024, 32768, "8", "vocab:0"),
    ]


def _log(rng, low, high, step):
    """A multiple of `step` from low to high, even over its logarithm."""
    return max(low, min(high, int(low * (high / low) ** rng.random()) // step * step))


def _split(rng, sizes):
    """A mesh of one or two dimensions and the tensor dimensions split over them, among those that the sizes allow: a batch dimension over the
    first mesh dimension, model dimensions over the other (the layouts of the paper)."""
    n_batch = rng.choice([n for n in (1, 1, 2, 4, 5, 8) if sizes["batch"] % n == 0])
    model = {k: v for k, v in sizes.items() if k != "batch"}
    n_model = rng.choice([1] + [n for n in (2, 4, 8, 16) if all(v % n == 0 and (v // n) % (1 if k == "heads" else 8) == 0 for k, v in model.items())])
    if n_batch == 1 and n_model == 1:
        return "1", ""
    if n_batch == 1:
        return str(n_model), ",".join("%s:0" % k for k in model)
    if n_model == 1:
        return str(n_batch), "batch:0"
    return "%dx%d" % (n_batch, n_model), ",".join(["batch:0"] + ["%s:1" % k for k in model])


def draw(rng):
    what = rng.choice(["ffn f32", "ffn", "ffn", "ffn", "attention", "attention", "attention", "decoder", "decoder", "vocab"])
    back = rng.random() < 0.75
    if what == "ffn f32":
        batch, d_model, d_ff = _log(rng, 4, 32, 1), _log(rng, 40, 512, 4), _log(rng, 72, 2048, 4)
        length = _log(rng, 1, 64, 1)
        while batch * length * d_model * d_ff > 8 * 128 * 256 * 1024:
            length = max(1, length // 2)
        return ffn("", "f32", batch, length, d_model, d_ff, *_split(rng, {"batch": batch, "d_ff": d_ff}), backward=back)
    if what == "ffn":
        batch, length, d_model, d_ff = _log(rng, 1, 64, 1), _log(rng, 24, 512, 1), _log(rng, 256, 2048, 8), _log(rng, 1024, 16384, 64)
        while batch * length * d_model * d_ff > 32 * 256 * 1024 * 32768:
            d_ff //= 2
        return ffn("", "bf16", batch, length, d_model, d_ff, *_split(rng, {"batch": batch, "d_ff": d_ff}), backward=back)
    d_k = rng.choice([64, 64, 64, 128])
    heads = rng.choice([4, 8, 16, 32]) * 64 // d_k
    if what == "attention":
        batch, length, d_model = _log(rng, 1, 32, 1), _log(rng, 40, 1536, 8), _log(rng, 256, 2048, 8)
        while batch * length > 16384 or batch * heads * length * length > 64 * 32 * 256 * 256:
            batch = max(1, batch // 2)
        return attention("", batch, length, d_model, heads, d_k, rng.random() < 0.6, *_split(rng, {"batch": batch, "heads": heads}), backward=back)
    if what == "decoder":
        batch, length, d_model, d_ff = _log(rng, 1, 64, 1), _log(rng, 40, 768, 8), _log(rng, 256, 2048, 8), _log(rng, 1024, 8192, 64)
        while batch * length > 16384 or batch * heads * length * length > 64 * 32 * 256 * 256:
            batch = max(1, batch // 2)
        return decoder("", batch, length, d_model, heads, d_k, d_ff, *_split(rng, {"batch": batch, "heads": heads, "d_ff": d_ff}), backward=back)
    batch, length, d_model, words = _log(rng, 1, 32, 1), _log(rng, 36, 256, 1), _log(rng, 128, 1024, 8), _log(rng, 1000, 32768, 8)
    return vocab("", batch, length, d_model, words, *_split(rng, {"batch": batch, "vocab": words}))


class _Inputs:
    """Seeded normal tensors on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, shape, dtype, scale=1.0, shift=0.0):
        t = torch.randn(shape, generator=self.g, device="cuda", dtype=torch.float32).mul_(scale).add_(shift)
        return t.to(dtype)

    def whole(self, high, n):
        return torch.randint(0, high, (n,), generator=self.g, device="cuda", dtype=torch.int32)


class _State:
    """What a program keeps from call to call: tensors, their named descriptors, the layout handle and the workspace."""

    def __init__(self, case):
        self.case, self.t, self.n, self.out = case, {}, {}, {}
        sizes = [int(s) for s in case["mesh"].split("x")]
        mesh = mtf.mtf_mesh_create([("mesh%d" % i, s) for i, s in enumerate(sizes)])
        rules = [r.split(":") for r in case["rules"].split(",") if r]
        self.layout = mtf.mtf_layout(mesh, [(d, "mesh" + m) for d, m in rules])

    def keep(self, name, t, dims, out=False):
        self.t[name], self.n[name] = t, mtf.named(t, dims)
        if out:
            self.out[name] = t

    def empty(self, name, shape, dims, dtype):
        self.keep(name, torch.empty(shape, dtype=dtype, device="cuda"), dims, out=True)

    def workspace(self, size):
        self.ws = torch.empty(size, dtype=torch.uint8, device="cuda")


def prepare(case, seed):
    r, s, kind = _Inputs(seed), _State(case), case["kind"]
    f32, bf = torch.float32, torch.bfloat16
    act = bf if case.get("dtype", "bf16") == "bf16" else f32
    B, L, D, back = case["batch"], case["length"], case["d_model"], case.get("backward", True)
    tok, words = ["batch", "length"], ["batch", "length", "d_model"]
    if kind == "vocab":
        V = case["vocab"]
        s.t["ids"], s.t["targets"] = r.whole(V, B * L), r.whole(V, B * L)
        for name, shape, dims, scale in (("table", (V, D), ["vocab", "d_model"], D ** -0.5), ("wout", (D, V), ["d_model", "vocab"], D ** -0.5)):
            master = r.normal(shape, f32, scale)
            s.keep(name, master.to(bf), dims, out=True)
            s.keep(name + "_master", master, dims, out=True)
            s.keep(name + "_momentum", torch.zeros_like(master), dims, out=True)
            s.empty("d" + name, shape, dims, f32)
        s.empty("x", (B, L, D), words, bf)
        s.empty("dx", (B, L, D), words, bf)
        s.empty("logits", (B, L, V), tok + ["vocab"], bf)
        s.empty("lse", (B, L), tok, f32)
        s.empty("loss", (B, L), tok, f32)
        s.keep("dloss", torch.full((B, L), 1.0 / (B * L), dtype=f32, device="cuda"), tok)
        parts = 16 * B * L * (V // 256 + 64)                    # the row statistics of mtf_xent_forward, for any split of the vocabulary
        sums = max(mtf.mtf_einsum_workspace_bytes(s.layout, [s.n["logits"], s.n["wout"]], s.n["dx"]),
                   mtf.mtf_einsum_workspace_bytes(s.layout, [s.n["x"], s.n["logits"]], s.n["dwout"]))
        s.workspace(max(parts, sums))
        return s
    x = r.normal((B, L, D), act)
    s.keep("x", x, words)
    if back:
        s.keep("dy", r.normal((B, L, D), act), words)
    params = {}
    if kind != "ffn":
        H, K = case["heads"], case["d_k"]
        for n in ("wq", "wk", "wv"):
            params[n] = (r.normal((D, H, K), bf, D ** -0.5), ["d_model", "heads", "d_v" if n == "wv" else "d_k"])
        params["wo"] = (r.normal((H, K, D), bf, (H * K) ** -0.5), ["heads", "d_v", "d_model"])
    if kind != "attention":
        F = case["d_ff"]
        params["w"] = (r.normal((D, F), act, D ** -0.5), ["d_model", "d_ff"])
        params["v"] = (r.normal((F, D), act, F ** -0.5), ["d_ff", "d_model"])
        params["bias"] = (r.normal((F,), f32, 0.1), ["d_ff"])
    if kind == "decoder":
        for n in ("ln1_gamma", "ln1_beta", "ln2_gamma", "ln2_beta"):
            params[n] = (r.normal((D,), f32, 0.1, 1.0 if "gamma" in n else 0.0), ["d_model"])
    for n, (t, dims) in params.items():
        s.keep(n, t, dims)
        if back:
            s.empty(GRADS[n], t.shape, dims, f32)
    saved = []
    if kind != "ffn":
        for n, shape, dims in (("q", (B, L, H, K), ["batch", "length", "heads", "d_k"]), ("kk", (B, L, H, K), ["batch", MEMORY, "heads", "d_k"]),
                               ("vv", (B, L, H, K), ["batch", MEMORY, "heads", "d_v"]), ("weights", (B, H, L, L), ["batch", "heads", "length", MEMORY]),
                               ("o", (B, L, H, K), ["batch", "length", "heads", "d_v"])):
            s.empty(n, shape, dims, bf)
            saved.append(n)
    if kind != "attention":
        s.empty("h", (B, L, F), tok + ["d_ff"], act)
        saved.append("h")
    if kind == "decoder":
        for n in ("s1", "a", "s2"):
            s.empty(n, (B, L, D), words, bf)
        for n in ("stats1", "stats2"):
            s.empty(n, (B, L, 2), tok + ["stat"], f32)
        saved += ["s1", "a", "s2", "stats1", "stats2"]
    s.empty("y", (B, L, D), words, act)
    if back:
        s.empty("dx", (B, L, D), words, act)
    s.params, s.saved = {n: s.n[n] for n in params}, {n: s.n[n] for n in saved}
    s.grads = {GRADS[n]: s.n[GRADS[n]] for n in params} if back else {}
    if kind == "ffn":
        s.workspace(mtf.mtf_ffn_workspace_bytes(s.layout, s.n["x"], s.n["w"]))
    elif kind == "attention":
        s.workspace(mtf.mtf_attention_workspace_bytes(s.layout, s.n["x"], s.n["wq"], s.n["wv"]))
    else:
        s.workspace(mtf.mtf_decoder_layer_workspace_bytes(s.layout, s.n["x"], s.params))
    return s


def run(s):
    n, lay, ws, kind = s.n, s.layout, s.ws, s.case["kind"]
    if kind == "vocab":
        mtf.mtf_embedding_forward(lay, s.t["ids"], n["table"], n["x"])
        mtf.mtf_xent_forward(lay, n["x"], n["wout"], s.t["targets"], n["logits"], n["lse"], n["loss"], ws)
        mtf.mtf_xent_backward(lay, n["x"], n["wout"], s.t["targets"], n["logits"], n["lse"], n["dloss"], n["dx"], n["dwout"], ws)
        mtf.mtf_embedding_backward(lay, s.t["ids"], n["dx"], n["dtable"])
        for w in ("table", "wout"):
            mtf.mtf_update(lay, n["d" + w], n[w + "_master"], n[w + "_momentum"], n[w], lr=0.01, momentum_coef=0.9, weight_decay=1e-4)
        return s.out
    back = s.case["backward"]
    if kind == "ffn":
        mtf.mtf_ffn_forward(lay, n["x"], n["w"], n["bias"], n["v"], n["h"], n["y"], ws)
        if back:
            mtf.mtf_ffn_backward(lay, n["x"], n["w"], n["v"], n["h"], n["dy"], n["dx"], n["dw"], n["dbias"], n["dv"], ws)
        return s.out
    causal = s.case["causal"]
    if kind == "attention":
        mtf.mtf_attention_forward(lay, n["x"], n["wq"], n["wk"], n["wv"], n["wo"], causal, None, n["q"], n["kk"], n["vv"], n["weights"], n["o"], n["y"], ws)
        if back:
            mtf.mtf_attention_backward(lay, n["x"], n["wq"], n["wk"], n["wv"], n["wo"], n["q"], n["kk"], n["vv"], n["weights"], n["o"], n["dy"], None, n["dx"],
                                       n["dwq"], n["dwk"], n["dwv"], n["dwo"], ws, causal=causal)
        return s.out
    mtf.mtf_decoder_layer_forward(lay, n["x"], s.params, causal, 1e-6, s.saved, n["y"], ws)
    if back:
        mtf.mtf_decoder_layer_backward(lay, n["x"], s.params, s.saved, n["dy"], n["dx"], s.grads, ws, causal=causal)
    return s.out


def work(case):
    B, L, D, kind = case["batch"], case["length"], case["d_model"], case["kind"]
    T, back = B * L, case.get("backward", True)
    passes, e = (3 if back else 1), (4 if case.get("dtype") == "f32" else 2)
    if kind == "vocab":
        V = case["vocab"]
        # ids and targets; x, its gradient and the logits (the entry points keep them); loss and lse; both tables: bf16 copy read and written,
        # master and momentum read and written, gradient written
        return {"bytes": T * (8 + 4 * D + 2 * V + 8) + 2 * V * D * (4 + 16 + 4), "flops": 6.0 * T * D * V}
    size = e * T * D * (4 if back else 2)                       # x and y, dy and dx
    flops = 0.0
    if kind != "ffn":
        H, K = case["heads"], case["d_k"]
        pairs = B * H * (L * (L + 1) // 2 if case["causal"] else L * L)
        size += 4 * D * H * K * (2 + (4 if back else 0)) + 4 * 2 * T * H * K + 2 * B * H * L * L
        flops += passes * (8.0 * T * D * H * K + 4.0 * pairs * K)
    if kind != "attention":
        F = case["d_ff"]
        size += 2 * D * F * (e + (4 if back else 0)) + 4 * F * (2 if back else 1) + e * T * F
        flops += passes * 4.0 * T * D * F
    if kind == "decoder":
        size += 2 * 3 * T * D + 16 * T + 16 * D * (2 if back else 1)
    return {"bytes": size, "flops": flops}


def tolerance(case):
    # Measured against the same blocks in 64 bits with the same intermediates rounded to bf16: 32 bits 5e-7 and at most 3e-6 of the rms; bf16 up to
    # 2e-3 (a sum that lands on the other side of a rounding step moves everything behind it) and at most 2.5e-2 of the rms.
    relu = "d_ff" in case
    if case.get("dtype") == "f32":
        hidden = case["batch"] * case["length"] * case["d_ff"]
        # a hidden unit within the rounding of its own sum (about 1e-7) of zero may fall on either side of the relu, which changes one of the
        # `hidden` elements of its gradient by its whole size: counted once there is a chance of it
        return {"rel": 1e-5, "max": 4e-5} if hidden < 100000 else {"rel": 1e-5 + 2.0 * hidden ** -0.5, "max": 0.5}
    return {"rel": 1e-2, "max": 0.5 if relu else 0.1}


def _attention_exact(x, p, heads_out, causal, scale):
    q, k, v = (torch.einsum("bld,dhk->blhk", x, p[n]) for n in ("wq", "wk", "wv"))
    s = torch.einsum("blhk,bmhk->bhlm", q, k).mul_(scale)
    if causal:
        s.masked_fill_(torch.ones(s.shape[-2:], dtype=torch.bool, device=s.device).triu(1), float("-inf"))
    w = torch.softmax(s, -1)
    o = torch.einsum("bhlm,bmhk->blhk", w, v)
    heads_out.update(q=q, kk=k, vv=v, weights=w, o=o)
    return torch.einsum("blhk,hkd->bld", o, p["wo"])


def _attention_grads(x, p, r, dy, scale):
    do = torch.einsum("bld,hkd->blhk", dy, p["wo"])
    r["dwo"] = torch.einsum("blhk,bld->hkd", r["o"], dy)
    dw = torch.einsum("blhk,bmhk->bhlm", do, r["vv"])
    dv = torch.einsum("bhlm,blhk->bmhk", r["weights"], do)
    ds = r["weights"] * (dw - (dw * r["weights"]).sum(-1, keepdim=True))
    dq, dk = (torch.einsum(e, ds, r[n]).mul_(scale) for e, n in (("bhlm,bmhk->blhk", "kk"), ("bhlm,blhk->bmhk", "q")))
    dx = 0.0
    for n, d in (("wq", dq), ("wk", dk), ("wv", dv)):
        r["d" + n] = torch.einsum("bld,blhk->dhk", x, d)
        dx = dx + torch.einsum("blhk,dhk->bld", d, p[n])
    return dx


def _ffn_exact(x, p, r):
    r["h"] = torch.relu(x @ p["w"] + p["bias"])
    return r["h"] @ p["v"]


def _ffn_grads(x, p, r, dy):
    dh = (dy @ p["v"].T) * (r["h"] > 0)
    r["dv"], r["dw"], r["dbias"] = r["h"].flatten(0, 1).T @ dy.flatten(0, 1), x.flatten(0, 1).T @ dh.flatten(0, 1), dh.sum((0, 1))
    return dh @ p["w"].T


def _norm_exact(x, gamma, beta):
    mu = x.mean(-1, keepdim=True)
    rstd = ((x - mu) ** 2).mean(-1, keepdim=True).add(1e-6).rsqrt()
    return gamma * (x - mu) * rstd + beta, torch.cat([mu, rstd], -1)


def _norm_grads(x, stats, gamma, dy):
    xh = (x - stats[..., :1]) * stats[..., 1:]
    g = dy * gamma
    dx = stats[..., 1:] * (g - g.mean(-1, keepdim=True) - xh * (g * xh).mean(-1, keepdim=True))
    return dx, (dy * xh).sum((0, 1)), dy.sum((0, 1))


def exact(case, seed):
    """What `run` returns, in 64 bits with nothing rounded in between, in plain torch."""
    s, kind, back = prepare(case, seed), case["kind"], case.get("backward", True)
    p = {n: t.double() if t.is_floating_point() else t.long() for n, t in s.t.items() if n not in s.out or kind == "vocab"}
    names = list(s.out)
    del s
    torch.cuda.empty_cache()
    r = {}
    if kind == "vocab":
        B, L = case["batch"], case["length"]
        x = p["table"][p["ids"]]
        z = x @ p["wout"]
        r["lse"] = torch.logsumexp(z, -1)
        r["loss"] = r["lse"] - z.gather(1, p["targets"][:, None])[:, 0]
        g = z.sub_(r["lse"][:, None]).exp_()
        g[torch.arange(B * L, device=g.device), p["targets"]] -= 1.0
        g.mul_(p["dloss"].view(-1, 1))
        r["logits"], r["x"], r["dx"], r["dwout"] = g, x, g @ p["wout"].T, x.T @ g
        r["dtable"] = torch.zeros_like(p["table"]).index_add_(0, p["ids"], r["dx"])
        for w in ("table", "wout"):
            r[w + "_momentum"] = 0.9 * p[w + "_momentum"] + r["d" + w]
            r[w + "_master"] = p[w + "_master"] - 0.01 * (r[w + "_momentum"] + 1e-4 * p[w + "_master"])
            r[w] = r[w + "_master"]
        for n in ("x", "dx", "logits", "lse", "loss"):
            r[n] = r[n].view(B, L, *r[n].shape[1:])
        return {n: r.get(n) for n in names}
    x, dy = p["x"], p.get("dy")
    if kind == "ffn":
        r["y"] = _ffn_exact(x, p, r)
        if back:
            r["dx"] = _ffn_grads(x, p, r, dy)
        return {n: r.get(n) for n in names}
    scale = case["d_k"] ** -0.5
    y = _attention_exact(x, p, r, case["causal"], scale)
    if kind == "attention":
        r["y"] = y
        if back:
            r["dx"] = _attention_grads(x, p, r, dy, scale)
        return {n: r.get(n) for n in names}
    r["s1"] = x + y
    r["a"], r["stats1"] = _norm_exact(r["s1"], p["ln1_gamma"], p["ln1_beta"])
    r["s2"] = r["a"] + _ffn_exact(r["a"], p, r)
    r["y"], r["stats2"] = _norm_exact(r["s2"], p["ln2_gamma"], p["ln2_beta"])
    if back:
        ds2, r["dln2_gamma"], r["dln2_beta"] = _norm_grads(r["s2"], r["stats2"], p["ln2_gamma"], dy)
        da = ds2 + _ffn_grads(r["a"], p, r, ds2)
        ds1, r["dln1_gamma"], r["dln1_beta"] = _norm_grads(r["s1"], r["stats1"], p["ln1_gamma"], da)
        r["dx"] = ds1 + _attention_grads(x, p, r, ds1, scale)
    return {n: r.get(n) for n in names}
