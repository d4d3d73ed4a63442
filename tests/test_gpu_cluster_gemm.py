"""bf16 contractions on 128-row tiles with K over a cluster, against the fp64 oracle.  The tests that ask for a variant run
every one (tiles of 64 and 128 columns, K over 1, 2, 4 and 8 CTAs) with operand orders, fused stages and column sums, and
check that it is the one that ran; the others take what the library chooses for few tiles and a longer and longer K."""
import contextlib

import numpy as np
import pytest

import seeded_inputs as si
from helpers import TOL, from_torch, parity_error, to_torch
from test_gpu_einsum import layout, mtf, run_einsum  # noqa: F401

pytestmark = pytest.mark.gpu

ONE = ([("all", 1)], [])
VARIANTS = [(columns, split) for columns in (64, 128) for split in (1, 2, 4, 8)]


@contextlib.contextmanager
def asked(mtf, variant):
    """Contractions inside run on this variant; the last of them is checked."""
    mtf.mtf_debug_contraction(*variant)
    try:
        yield
    finally:
        ran = mtf.mtf_debug_contraction(0, 0)
    assert ran == variant


@pytest.mark.parametrize("variant", VARIANTS, ids=str)
@pytest.mark.parametrize("order", ["ik,kj", "ik,jk", "ki,kj", "ki,jk"])
def test_every_variant(mtf, variant, order):
    for m, n, k in ((8, 8, 520), (136, 200, 1032), (264, 72, 512)):
        size = {"i": m, "j": n, "k": k}
        a, b = [[(c, size[c]) for c in t] for t in order.split(",")]
        for dt in ("bf16", "f32"):
            with asked(mtf, variant):
                got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), [a, b], [("i", m), ("j", n)], "bf16", dt)
            assert parity_error(got, ref) <= TOL["bf16"]


@pytest.mark.parametrize("variant", VARIANTS, ids=str)
@pytest.mark.parametrize("out_dtype", ["bf16", "f32"])
def test_every_variant_with_stages(mtf, variant, out_dtype):
    size = {"i": 264, "j": 136, "k": 1032}
    dims = [[(c, size[c]) for c in t] for t in ("ik", "kj")]
    for out in ("ij", "ji"):
        for bias in "ij":
            ep = {"scale": -0.5, "bias": [(bias, size[bias])], "relu": True, "relu_mask": True, "residual": True}
            with asked(mtf, variant):
                got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), dims, [(c, size[c]) for c in out], "bf16", out_dtype, epilogue=ep)
            assert parity_error(got, ref) <= TOL["bf16"]


@pytest.mark.parametrize("variant", VARIANTS, ids=str)
@pytest.mark.parametrize("m", [8, 100, 300])
def test_every_variant_with_column_sums(mtf, variant, m):
    """One block of rows: stored by its CTA or gathered inside the cluster; several: partial rows in the workspace, or atomics
    without one.  All but the last repeat bit for bit."""
    import torch
    n, k = 136, 1032
    x, y, mask = si.normal(3, "x", [m, k], "bf16"), si.normal(3, "y", [k, n], "bf16", k ** -0.5), si.normal(3, "mask", [m, n], "bf16")
    tx, ty, tm, lay = to_torch(x), to_torch(y), to_torch(mask), layout(mtf, *ONE)
    ref = ((x.f64 @ y.f64) * (mask.f64 > 0)).sum(0)
    for scratch in (0, 1 << 20):
        ws = torch.empty(scratch, dtype=torch.uint8, device="cuda") if scratch else None
        cols = [torch.full((n,), float("nan"), device="cuda") for _ in range(5)]
        for col in cols:
            out = torch.empty(m, n, dtype=torch.bfloat16, device="cuda")
            ep = mtf.Epilogue(relu_mask=mtf.named(tm, ["i", "j"]), reduce_sum_out=mtf.named(col, ["j"]))
            with asked(mtf, variant):
                mtf.mtf_einsum(lay, None, [mtf.named(tx, ["i", "k"]), mtf.named(ty, ["k", "j"])], mtf.named(out, ["i", "j"]), ep, ws)
        mtf.mtf_device_status()
        assert parity_error(from_torch(cols[0]), ref) <= TOL["f32"]
        if scratch or m <= 128:
            assert all(torch.equal(cols[0], c) for c in cols[1:])


@pytest.mark.parametrize("m,n,k", [(8, 8, 8), (128, 64, 64), (136, 72, 640), (40, 200, 1024), (264, 56, 1096), (24, 72, 4096)])
@pytest.mark.parametrize("order", ["ik,kj", "ik,jk", "ki,kj", "ki,jk"])
def test_orders_edges_and_splits(mtf, order, m, n, k):
    size = {"i": m, "j": n, "k": k}
    a, b = [[(c, size[c]) for c in t] for t in order.split(",")]
    for out, dt in ((["i", "j"], "bf16"), (["i", "j"], "f32"), (["j", "i"], "bf16")):
        got, ref, info = run_einsum(mtf, layout(mtf, *ONE), [a, b], [(c, size[c]) for c in out], "bf16", dt)
        assert info["kernel_kind"] == mtf.MTF_KERNEL_TCGEN05
        assert parity_error(got, ref) <= TOL["bf16"]


def test_wider_tiles(mtf):
    a, b = [("b", 200), ("i", 41), ("k", 72)], [("b", 200), ("k", 72), ("j", 136)]
    got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), [a, b], [("b", 200), ("i", 41), ("j", 136)], "bf16")
    assert parity_error(got, ref) <= TOL["bf16"]
    a, b = [("k", 4096), ("i", 1000)], [("k", 4096), ("j", 1032)]
    got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), [a, b], [("i", 1000), ("j", 1032)], "bf16", "f32")
    assert parity_error(got, ref) <= TOL["bf16"]


@pytest.mark.parametrize("mesh,rules", [ONE, ([("r", 5), ("c", 4)], [("b", "r"), ("k", "c")])], ids=["whole", "split"])
def test_batch_dims_and_slices(mtf, mesh, rules):
    a, b = [("b", 5), ("l", 37), ("h", 3), ("k", 64)], [("b", 5), ("m", 40), ("h", 3), ("k", 64)]
    got, ref, _ = run_einsum(mtf, layout(mtf, mesh, rules), [a, b], [("b", 5), ("h", 3), ("l", 37), ("m", 40)], "bf16", "f32")
    assert parity_error(got, ref) <= TOL["bf16"]
    a, b = [("b", 5), ("l", 37), ("k", 256)], [("k", 256), ("j", 104)]
    got, ref, _ = run_einsum(mtf, layout(mtf, mesh, rules), [a, b], [("b", 5), ("l", 37), ("j", 104)], "bf16")
    assert parity_error(got, ref) <= TOL["bf16"]


@pytest.mark.parametrize("m,n,k", [(136, 72, 64), (100, 136, 640), (264, 64, 1024), (24, 72, 4096)])
@pytest.mark.parametrize("out_dtype", ["bf16", "f32"])
@pytest.mark.parametrize("out", [["i", "j"], ["j", "i"]], ids=["in-order", "exchanged"])
def test_stages(mtf, out, out_dtype, m, n, k):
    size = {"i": m, "j": n, "k": k}
    if out[1] == "i":
        size["i"] = (m + 7) // 8 * 8                  # (the contiguous output dimension holds whole store pieces)
    dims = [[(c, size[c]) for c in t] for t in ("ik", "kj")]
    for bias in ("i", "j"):
        ep = {"scale": -0.5, "bias": [(bias, size[bias])], "relu": True, "relu_mask": True, "residual": True}
        got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), dims, [(c, size[c]) for c in out], "bf16", out_dtype, epilogue=ep)
        assert parity_error(got, ref) <= TOL["bf16"]


@pytest.mark.parametrize("m,n,k", [(8, 72, 64), (300, 136, 640), (136, 64, 4096)])
@pytest.mark.parametrize("scratch", [0, 1 << 22])
def test_column_sums(mtf, scratch, m, n, k):
    import torch
    x, y = si.normal(3, "x", [m, k], "bf16"), si.normal(3, "y", [k, n], "bf16", k ** -0.5)
    mask = si.normal(3, "mask", [m, n], "bf16")
    out, col = torch.full((m, n), float("nan"), dtype=torch.bfloat16, device="cuda"), torch.full((n,), float("nan"), device="cuda")
    ep = mtf.Epilogue(relu_mask=mtf.named(to_torch(mask), ["i", "j"]), reduce_sum_out=mtf.named(col, ["j"]))
    ws = torch.empty(scratch, dtype=torch.uint8, device="cuda") if scratch else None
    mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(to_torch(x), ["i", "k"]), mtf.named(to_torch(y), ["k", "j"])], mtf.named(out, ["i", "j"]), ep, ws)
    mtf.mtf_device_status()
    ref = (x.f64 @ y.f64) * (mask.f64 > 0)
    assert parity_error(from_torch(out), ref) <= TOL["bf16"]
    assert parity_error(from_torch(col), ref.sum(0)) <= TOL["f32"]


@pytest.mark.parametrize("m", [8, 24, 136, 200])
@pytest.mark.parametrize("k", [256, 640, 4096])
def test_tiles_with_few_rows_leave_the_cluster_together(mtf, m, k):
    """Most CTAs of a cluster own no row of such a tile (or of the last one): launches back to back, more than fill the chip,
    all give the first one's bits."""
    import torch
    n = 1032
    x, y = si.normal(7, "x", [m, k], "bf16"), si.normal(7, "y", [k, n], "bf16", k ** -0.5)
    tx, ty, lay = to_torch(x), to_torch(y), layout(mtf, *ONE)
    outs = [torch.full((m, n), float("nan"), device="cuda") for _ in range(40)]
    for out in outs:
        mtf.mtf_einsum(lay, None, [mtf.named(tx, ["i", "k"]), mtf.named(ty, ["k", "j"])], mtf.named(out, ["i", "j"]))
    mtf.mtf_device_status()
    assert parity_error(from_torch(outs[0]), x.f64 @ y.f64) <= TOL["bf16"]
    assert all(torch.equal(outs[0], o) for o in outs[1:])


@pytest.mark.parametrize("m,n,k,split", [(200, 512, 2048, 8), (136, 64, 4096, 8), (300, 136, 640, 2)])
@pytest.mark.parametrize("room", ["reported", "a row per 32 rows"])
def test_column_sums_repeat_with_the_reported_workspace(mtf, m, n, k, split, room):
    """... and with one of a partial row per 32 rows, the persistent kernel's, which holds those of a split of 4."""
    import torch
    x, y = si.normal(3, "x", [m, k], "bf16"), si.normal(3, "y", [k, n], "bf16", k ** -0.5)
    tx, ty, lay = to_torch(x), to_torch(y), layout(mtf, *ONE)
    nx, ny = mtf.named(tx, ["i", "k"]), mtf.named(ty, ["k", "j"])
    cols = [torch.full((n,), float("nan"), device="cuda") for _ in range(20)]
    for col in cols:
        out = mtf.named(torch.empty(m, n, dtype=torch.bfloat16, device="cuda"), ["i", "j"])
        ep = mtf.Epilogue(relu=True, reduce_sum_out=mtf.named(col, ["j"]))
        size = mtf.mtf_einsum_workspace_bytes(lay, [nx, ny], out, ep)
        if room != "reported":
            size = (m + 127) // 128 * 4 * n * 4
        mtf.mtf_einsum(lay, None, [nx, ny], out, ep, torch.empty(size, dtype=torch.uint8, device="cuda"))
    mtf.mtf_device_status()
    assert mtf.mtf_debug_contraction()[1] == (split if room == "reported" else min(split, 4))
    assert parity_error(from_torch(cols[0]), np.maximum(x.f64 @ y.f64, 0).sum(0)) <= TOL["f32"]
    assert all(torch.equal(cols[0], c) for c in cols[1:])


# which side of the rule a product lies on: few tiles on the cluster kernel; a chip full of 128-row tiles, where rows off
# 128-byte lines and f32 outputs measured 1.15 to 1.5 times their time on the persistent kernel, there
@pytest.mark.parametrize("a,b,out,dtype,cluster", [
    ([128, 4096], [4096, 1024], [128, 1024], "bf16", True), ([512, 1024], [1024, 1024], [512, 1024], "bf16", True),
    ([2664, 200], [2992, 200], [2664, 2992], "f32", False), ([264, 3032], [264, 1792], [3032, 1792], "bf16", False),
    ([2160, 264], [3176, 264], [2160, 3176], "f32", False), ([6208, 112], [112, 944], [6208, 944], "f32", False)])
def test_which_products_it_takes(mtf, a, b, out, dtype, cluster):
    import torch
    k = (set(a) & set(b)).pop()
    sizes = [dict(zip(("i", "k") if a[1] == k else ("k", "i"), a)), dict(zip(("k", "j") if b[0] == k else ("j", "k"), b))]
    t = [torch.randn(list(s.values()), device="cuda").to(torch.bfloat16) for s in sizes]
    c = torch.empty(out, dtype=torch.float32 if dtype == "f32" else torch.bfloat16, device="cuda")
    mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(x, list(s)) for x, s in zip(t, sizes)], mtf.named(c, ["i", "j"]))
    mtf.mtf_device_status()
    assert (mtf.mtf_debug_contraction()[1] > 0) == cluster


@pytest.mark.parametrize("n", [8, 64, 68, 72, 136, 200])
@pytest.mark.parametrize("shift", [0, 4])
@pytest.mark.parametrize("columns,split", [(64, 1), (64, 4), (128, 1), (128, 2)])
def test_f32_rows_on_and_off_32_bytes(mtf, n, shift, columns, split):
    """f32 results are stored 32 bytes at a time where every row starts on 32 bytes, else 16: row lengths of either kind, outputs that start on 16 bytes only."""
    import torch
    m, k = 200, 264
    g = torch.Generator(device="cuda").manual_seed(2)
    x, y = torch.randn(m, k, generator=g, device="cuda").bfloat16(), torch.randn(n, k, generator=g, device="cuda").bfloat16()      # (B along K: any n)
    room = torch.full((m * n + 16,), 7.0, device="cuda")
    out = room[shift:shift + m * n].view(m, n)
    mtf.mtf_debug_contraction(columns, split)
    try:
        mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(x, ["i", "k"]), mtf.named(y, ["j", "k"])], mtf.named(out, ["i", "j"]))
    finally:
        assert mtf.mtf_debug_contraction(0, 0) == (columns, split)
    mtf.mtf_device_status()
    ref = x.double() @ y.double().t()
    # f32 sums of k products, of which the accumulator drops at most 2^-23 of the running sum each
    assert ((out.double() - ref).abs() / ref.abs().clamp_min(k ** 0.5)).max() <= k * 2.0 ** -23
    assert (room[:shift] == 7.0).all() and (room[shift + m * n:] == 7.0).all()
