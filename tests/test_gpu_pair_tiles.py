"""The tiles that CTA pairs may take beside 256 columns inside a slice: 192 columns (an N-contiguous B in 32-column boxes) and 128, and tiles across the edges of
slices.  Sizes at which the launcher's estimate takes each, whole and ragged, with every operand order and fused stage, against 64-bit sums."""
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
