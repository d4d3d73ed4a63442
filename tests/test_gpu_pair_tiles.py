"""The tiles that CTA pairs may take beside 256 columns inside a slice: 192 columns (an N-contiguous B in 32-column boxes) and 128, and tiles across the edges of
slices, whole and ragged, with every operand order and fused stage, against 64-bit sums.  The first test leaves the tiles to the launcher's estimate, the others
ask for each by name or look at what the estimate took."""
import pytest

from test_gpu_einsum import layout, mtf  # noqa: F401

pytestmark = pytest.mark.gpu

# (batch, m, n, k, slices of m): nine batches of two row tiles fill the 74 pairs once with four 192-column tiles of 768 columns and twice with six of 128; few
# tiles take 128 columns; five slices of 333 rows are ten tiles of 256 rows, seven across their edges
SHAPES = [(9, 512, 768, 320, 1), (9, 500, 760, 328, 1), (9, 512, 576, 64, 1), (1, 512, 512, 256, 1), (1, 264, 136, 72, 1), (1, 1665, 776, 200, 5), (1, 1665, 3080, 200, 5)]


@pytest.mark.parametrize("b,m,n,k,slices", SHAPES)
@pytest.mark.parametrize("order", ["ik,kj", "ik,jk", "ki,kj", "ki,jk"])
@pytest.mark.parametrize("stage", ["plain", "f32", "bias relu", "mask sums", "residual"])
def test_narrow_tiles_and_tiles_across_slices(mtf, b, m, n, k, slices, order, stage):  # noqa: F811
    import torch
    if "ki" in order and (m // slices) % 8:
        pytest.skip("slices of a row-contiguous operand start on 16 bytes")
    if b > 1 and stage == "mask sums":
        b = 1                       # (a batched output keeps no fused column sums)
    g = torch.Generator(device="cuda").manual_seed(1)
    size = {"i": m, "j": n, "k": k}
    a_order, b_order = order.split(",")
    A, B = [torch.randn(b, *[size[c] for c in o], generator=g, device="cuda").bfloat16() for o in (a_order, b_order)]
    out = torch.full((b, m, n), float("nan"), device="cuda", dtype=torch.float32 if stage == "f32" else torch.bfloat16)
    ref = torch.einsum("b%s,b%s->bij" % (a_order, b_order), A.double(), B.double())
    one = b == 1
    named = lambda t, names: mtf.named(t[0] if one else t, names if one else ["b"] + names)  # noqa: E731
    no, keep, kw, sums = named(out, ["i", "j"]), [], {}, None
    if stage == "bias relu":
        bias = torch.randn(n, generator=g, device="cuda")
        ref = (ref + bias.double()).relu()
        kw, keep = {"bias": mtf.named(bias, ["j"]), "relu": True}, [bias]
    elif stage == "mask sums":
        mask, sums = torch.randn(b, m, n, generator=g, device="cuda").bfloat16(), torch.full((n,), float("nan"), device="cuda")
        ref = ref * (mask.double() > 0)
        kw, keep = {"relu_mask": named(mask, ["i", "j"]), "reduce_sum_out": mtf.named(sums, ["j"])}, [mask]
    elif stage == "residual":
        r = torch.randn(b, m, n, generator=g, device="cuda").bfloat16()
        ref = ref + r.double()
        kw, keep = {"residual": named(r, ["i", "j"])}, [r]
    ep = mtf.Epilogue(**kw) if kw else None
    mtf.mtf_plan_force(1, -1)       # CTA pairs, whose tiles the launcher chooses
    try:
        lay = layout(mtf, [("p", slices)], [("i", "p")] if slices > 1 else [])
        ins = [named(A, list(a_order)), named(B, list(b_order))]
        ws = torch.empty(max(256, mtf.mtf_einsum_workspace_bytes(lay, ins, no, ep)), dtype=torch.uint8, device="cuda")
        mtf.mtf_einsum(lay, None, ins, no, ep, ws)
    finally:
        mtf.mtf_plan_force(-1, -1)
    mtf.mtf_device_status()
    # one rounding to the stored type, and f32 sums of k products of which the accumulator drops at most 2^-23 of the running sum each
    scale = ref.abs().clamp_min((k ** 0.5))
    assert ((out.double() - ref).abs() / scale).max() <= (2.0 ** -8 if stage != "f32" else 0.0) + k * 2.0 ** -23
    if sums is not None:
        assert ((sums.double() - ref.sum((0, 1))).abs() / (m * k) ** 0.5).max() <= 1e-4


# ---- each tile by name: columns x inside or across the slices, at sizes where rows, columns, both and neither are split and no tile divides a slice ----------
SPLIT = [(624, 1160, 136, 2, 1), (520, 1160, 136, 1, 5), (624, 1160, 200, 2, 5), (264, 136, 72, 1, 1), (304, 640, 64, 1, 1)]


def product(mtf, m, n, k, sm, sn, order, stage, tiles):  # noqa: F811
    """(device outputs, fp64 references, tiles that ran) of one product on CTA pairs."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(2)
    size = {"i": m, "j": n, "k": k}
    a_order, b_order = order.split(",")
    A, B = [torch.randn(*[size[c] for c in o], generator=g, device="cuda").bfloat16() for o in (a_order, b_order)]
    out = torch.full((m, n), float("nan"), device="cuda", dtype=torch.float32 if stage == "f32" else torch.bfloat16)
    ref = torch.einsum("%s,%s->ij" % (a_order, b_order), A.double(), B.double())
    kw, sums = {}, None
    if stage == "bias relu":
        bias = torch.randn(n, generator=g, device="cuda")
        ref, kw = (ref + bias.double()).relu(), {"bias": mtf.named(bias, ["j"]), "relu": True}
    elif stage == "mask sums":
        mask, sums = torch.randn(m, n, generator=g, device="cuda").bfloat16(), torch.full((n,), float("nan"), device="cuda")
        ref, kw = ref * (mask.double() > 0), {"relu_mask": mtf.named(mask, ["i", "j"]), "reduce_sum_out": mtf.named(sums, ["j"])}
    elif stage == "residual":
        r = torch.randn(m, n, generator=g, device="cuda").bfloat16()
        ref, kw = ref + r.double(), {"residual": mtf.named(r, ["i", "j"])}
    ep = mtf.Epilogue(**kw) if kw else None
    lay = layout(mtf, [("r", sm), ("c", sn)], [d for d, s in (("i", sm), ("j", sn)) if s > 1 for d in [(d, "r" if d == "i" else "c")]])
    ins, no = [mtf.named(A, list(a_order)), mtf.named(B, list(b_order))], mtf.named(out, ["i", "j"])
    mtf.mtf_plan_force(1, -1)
    mtf.mtf_debug_pair_tiles(*tiles)
    try:
        ws = torch.empty(max(256, mtf.mtf_einsum_workspace_bytes(lay, ins, no, ep)), dtype=torch.uint8, device="cuda")
        mtf.mtf_einsum(lay, None, ins, no, ep, ws)
    finally:
        mtf.mtf_plan_force(-1, -1)
        ran = mtf.mtf_debug_pair_tiles(0)
    mtf.mtf_device_status()
    return out, sums, ref, ran


@pytest.mark.parametrize("m,n,k,sm,sn", SPLIT)
@pytest.mark.parametrize("order", ["ik,kj", "ik,jk", "ki,kj", "ki,jk"])
@pytest.mark.parametrize("stage", ["plain", "f32", "bias relu", "mask sums", "residual"])
@pytest.mark.parametrize("columns", [128, 192, 256])
@pytest.mark.parametrize("across", [False, True])
def test_the_tiles_that_are_asked_for(mtf, m, n, k, sm, sn, order, stage, columns, across):  # noqa: F811
    if sm * sn == 1 and across:
        pytest.skip("one slice has no edges to cross")
    out, sums, ref, ran = product(mtf, m, n, k, sm, sn, order, stage, (columns, across))
    assert ran == (columns, across)
    # (as above: one rounding to the stored type, f32 sums of k products)
    scale = ref.abs().clamp_min(k ** 0.5)
    assert ((out.double() - ref).abs() / scale).max() <= (2.0 ** -8 if stage != "f32" else 0.0) + k * 2.0 ** -23
    if sums is not None:
        assert ((sums.double() - ref.sum(0)).abs() / (m * k) ** 0.5).max() <= 1e-4


def test_what_may_not_choose_keeps_256_columns(mtf):  # noqa: F811
    """A forced reduce mode leaves the tiles alone, whatever is asked for."""
    import torch
    lay = layout(mtf, [("p", 2)], [("k", "p")])
    a, b, c = (torch.randn(*s, device="cuda").bfloat16() for s in ((512, 256), (256, 512), (512, 512)))
    mtf.mtf_plan_force(1, 1)
    mtf.mtf_debug_pair_tiles(128)
    try:
        mtf.mtf_einsum(lay, None, [mtf.named(a, ["i", "k"]), mtf.named(b, ["k", "j"])], mtf.named(c, ["i", "j"]), None, None)
    finally:
        mtf.mtf_plan_force(-1, -1)
        ran = mtf.mtf_debug_pair_tiles(0)
    assert ran == (256, False)


# (sizes of the ragged feed-forward block and of the first test; columns and whether tiles cross the slices)
@pytest.mark.parametrize("b,m,n,k,slices,order,want", [(1, 2048, 2048, 512, 1, "ik,kj", (256, False)), (9, 512, 768, 320, 1, "ik,kj", (192, False)), (9, 512, 768, 320, 1, "ik,jk", (192, False)),
                                                       (1, 512, 512, 256, 1, "ik,kj", (128, False)), (1, 1665, 3080, 776, 5, "ik,jk", (192, True)), (1, 1640, 1280, 2048, 5, "ik,kj", (128, True)), (1, 1640, 2560, 512, 5, "ik,jk", (256, True))])
def test_the_estimate_takes_every_kind(mtf, b, m, n, k, slices, order, want):  # noqa: F811
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the estimate counts waves of 148 SMs")
    size = {"i": m, "j": n, "k": k}
    named = lambda names: mtf.named(torch.zeros(*([b] if b > 1 else []), *[size[c] for c in names], dtype=torch.bfloat16, device="cuda"), (["b"] if b > 1 else []) + list(names))  # noqa: E731
    mtf.mtf_plan_force(1, -1)
    try:
        mtf.mtf_einsum(layout(mtf, [("p", slices)], [("i", "p")] if slices > 1 else []), None, [named(o) for o in order.split(",")], named("ij"), None, None)
    finally:
        mtf.mtf_plan_force(-1, -1)
    mtf.mtf_device_status()
    assert mtf.mtf_debug_pair_tiles(0) == want


@pytest.mark.parametrize("columns", [128, 192])
def test_grouped_and_three_term_launches(mtf, columns):  # noqa: F811
    """The weight gradients of attention (one grouped launch) and dx (three products in one accumulator): a sum over K does not depend on the tile, so the bits
    are those of 256 columns."""
    import torch
    B, L, M, H, K = 3, 200, 520, 8, 64
    g = torch.Generator(device="cuda").manual_seed(5)
    words, f32 = ["batch", "length", "d_model"], torch.float32
    shapes = {"x": ((B, L, M), words), "dy": ((B, L, M), words), "dx": ((B, L, M), words), "y": ((B, L, M), words), "weights": ((B, H, L, L), ["batch", "heads", "length", "memory_length"])}
    for w in ("wq", "wk", "wv"):
        shapes[w] = shapes["d" + w] = ((M, H, K), ["d_model", "heads", "d_v" if w == "wv" else "d_k"])
    shapes["wo"] = shapes["dwo"] = ((H, K, M), ["heads", "d_v", "d_model"])
    for a in ("q", "kk", "vv", "o"):
        shapes[a] = ((B, L, H, K), ["batch", "length" if a in ("q", "o") else "memory_length", "heads", "d_v" if a in ("vv", "o") else "d_k"])
    t = {k: (torch.randn(*s, generator=g, device="cuda") * (M ** -0.5 if k[0] == "w" and k != "weights" else 1.0)).to(f32 if k[:2] == "dw" else torch.bfloat16)
         for k, (s, _) in shapes.items()}
    n = {k: mtf.named(t[k], d) for k, (_, d) in shapes.items()}
    lay = layout(mtf, [("p", 2)], [("heads", "p")])
    ws = torch.empty(mtf.mtf_attention_workspace_bytes(lay, n["x"], n["wq"], n["wv"]), dtype=torch.uint8, device="cuda")
    mtf.mtf_attention_forward(lay, *[n[k] for k in ("x", "wq", "wk", "wv", "wo")], True, None, *[n[k] for k in ("q", "kk", "vv", "weights", "o", "y")], ws)
    got = []
    for tiles in ((256, False), (columns, False), (columns, True)):
        mtf.mtf_plan_force(1, -1)
        mtf.mtf_debug_pair_tiles(*tiles)
        try:
            mtf.mtf_attention_backward(lay, *[n[k] for k in ("x", "wq", "wk", "wv", "wo", "q", "kk", "vv", "weights", "o", "dy")], None,
                                       *[n[k] for k in ("dx", "dwq", "dwk", "dwv", "dwo")], ws, causal=True)
        finally:
            mtf.mtf_plan_force(-1, -1)
            ran = mtf.mtf_debug_pair_tiles(0)
        mtf.mtf_device_status()
        assert ran[0] == tiles[0], (ran, tiles)          # (dx; the weight gradients' plan may choose under the same conditions)
        got.append([t[k].clone() for k in ("dx", "dwq", "dwk", "dwv", "dwo")])
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0], other))
