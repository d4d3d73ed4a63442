"""The f32 products that run on the tensor cores in bf16 pieces: edges of the 128 x 64 tile, of the 64-deep stage and its 16-deep
steps, every split of K, operand orders, the fused stages, values whose pieces leave bf16's range, and the error
against 64 bits beside that of plain FP32 arithmetic."""
import numpy as np
import pytest

from helpers import TOL, from_torch, parity_error
from test_gpu_einsum import layout, mtf, run_einsum  # noqa: F401

pytestmark = pytest.mark.gpu
ONE = ([("all", 1)], [])


@pytest.fixture
def asked(mtf):  # noqa: F811
    mtf.mtf_debug_contraction(128, 1)
    yield
    assert mtf.mtf_debug_contraction(0, 0)[0] == 128


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (128, 64, 64), (129, 65, 65), (127, 63, 16), (5, 200, 17), (260, 36, 1000), (8, 64, 33), (1000, 520, 130)])
@pytest.mark.parametrize("order", ["ik,kj", "ik,jk", "ki,kj", "ki,jk"])
def test_orders_and_edges(mtf, asked, order, m, n, k):  # noqa: F811
    size = {"i": m, "j": n, "k": k}
    a, b = [[(c, size[c]) for c in t] for t in order.split(",")]
    for out, dt in ((["i", "j"], "f32"), (["j", "i"], "f32"), (["i", "j"], "bf16")):
        got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), [a, b], [(c, size[c]) for c in out], "f32", dt)
        assert parity_error(got, ref) <= TOL[dt]


@pytest.mark.parametrize("m,n,k", [(8, 256, 64), (77, 101, 300), (520, 130, 64)])
def test_stages_and_column_sums(mtf, asked, m, n, k):  # noqa: F811
    import torch
    size = {"i": m, "j": n, "k": k}
    dims = [[(c, size[c]) for c in t] for t in ("ik", "kj")]
    for out in ("ij", "ji"):
        for bias in "ij":
            ep = {"scale": -0.5, "bias": [(bias, size[bias])], "relu": True, "relu_mask": True, "residual": True}
            got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), dims, [(c, size[c]) for c in out], "f32", epilogue=ep)
            assert parity_error(got, ref) <= TOL["f32"]
    x, y = torch.randn(m, k, device="cuda"), torch.randn(k, n, device="cuda")
    o, col = torch.empty(m, n, device="cuda"), torch.full((n,), float("nan"), device="cuda")
    mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(x, ["i", "k"]), mtf.named(y, ["k", "j"])], mtf.named(o, ["i", "j"]),
                   mtf.Epilogue(relu=True, reduce_sum_out=mtf.named(col, ["j"])))
    assert parity_error(from_torch(col), (x.double() @ y.double()).relu().sum(0).cpu().numpy()) <= TOL["f32"]


@pytest.mark.parametrize("m,n,k", [(130, 70, 70), (33, 65, 300), (128, 64, 256)])
@pytest.mark.parametrize("dims", ["bihk,bjhk,bhij", "bihk,bhkj,bihj", "bhki,bkhj,bhji", "hbik,bhkj,bihj", "bik,bkj,bji", "kbi,jbk,bij"])
def test_batches(mtf, asked, dims, m, n, k):  # noqa: F811
    """One and two batch dimensions beside and between the others, row lengths and batch strides on and off 16 bytes, operands exchanged."""
    size = {"b": 2, "h": 3, "i": m, "j": n, "k": k}
    a, b, out = [[(c, size[c]) for c in t] for t in dims.split(",")]
    for dt in ("f32", "bf16"):
        got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), [a, b], out, "f32", dt)
        assert parity_error(got, ref) <= TOL[dt]
    ep = {"scale": 2.0, "bias": [("j", n)], "relu": True, "residual": True}
    got, ref, _ = run_einsum(mtf, layout(mtf, *ONE), [a, b], out, "f32", epilogue=ep)
    assert parity_error(got, ref) <= TOL["f32"]


@pytest.mark.parametrize("batch,m,n,k,split", [(1, 300, 70, 70, 2), (1, 2100, 70, 20, 1), (3, 40, 70, 300, 4), (1, 40, 70, 300, 4)])
def test_column_sums_over_tiles_and_batches(mtf, asked, batch, m, n, k, split):  # noqa: F811
    """Sums over every row of every batch entry: several row tiles add to the zeroed output, one row tile stores it, a cluster gathers it."""
    import torch
    x, y = torch.randn(batch, m, k, device="cuda"), torch.randn(batch, k, n, device="cuda")
    o, col = torch.empty(batch, m, n, device="cuda"), torch.full((n,), float("nan"), device="cuda")
    mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(x, ["b", "i", "k"]), mtf.named(y, ["b", "k", "j"])], mtf.named(o, ["b", "i", "j"]),
                   mtf.Epilogue(reduce_sum_out=mtf.named(col, ["j"])))
    assert mtf.mtf_debug_contraction(128, 1) == (128, split)
    ref = x.double() @ y.double()
    assert parity_error(from_torch(o), ref.cpu().numpy()) <= TOL["f32"]
    assert parity_error(from_torch(col), ref.sum((0, 1)).cpu().numpy()) <= TOL["f32"]


def product(mtf, x, y, columns):  # noqa: F811
    import torch
    o = torch.full((x.shape[0], y.shape[1]), float("nan"), device="cuda")
    mtf.mtf_debug_contraction(columns, 1)
    mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(x, ["i", "k"]), mtf.named(y, ["k", "j"])], mtf.named(o, ["i", "j"]))
    assert mtf.mtf_debug_contraction(0, 0)[0] == columns
    mtf.mtf_device_status()
    return o


@pytest.mark.parametrize("k", [16, 64, 256, 1000, 4096])
def test_error_is_no_larger_than_plain_arithmetic(mtf, k):  # noqa: F811
    """Both within a few roundings of the sum; the pieces' rounding is below that of one chain of f32 additions."""
    import torch
    torch.manual_seed(k)
    x, y = torch.randn(384, k, device="cuda"), torch.randn(k, 192, device="cuda")
    ref = x.double() @ y.double()
    err = [((product(mtf, x, y, c).double() - ref).norm() / ref.norm()).item() for c in (64, 128)]
    assert err[1] <= err[0]


@pytest.mark.parametrize("k", [40, 520])
def test_values_outside_the_pieces_range(mtf, k):  # noqa: F811
    """Infinities, NaN and the type's largest values come out as plain f32 arithmetic has them, and so do small values beside ordinary and small ones."""
    import torch
    torch.manual_seed(1)
    x, y = torch.randn(200, k, device="cuda"), torch.randn(k, 100, device="cuda")
    x[3, 5], x[17, 0], x[40, k - 1], x[41, 7] = float("inf"), float("nan"), -float("inf"), float("inf")
    x[60] = torch.where(torch.arange(k, device="cuda") % 2 == 0, 3.4e38, 0.0)      # rounds to infinity as a bf16
    y[:, 9] = 0.0                                                                       # infinity times zero
    y[:, 10] = torch.where(torch.arange(k, device="cuda") == 0, 0.5, 0.0)
    x[90] = float(np.finfo(np.float32).min)
    y[:, 11] = 0.0
    y[2, 11] = 1.0
    x[100] *= 1e-36
    y[:, 20] *= 1e-37
    got = product(mtf, x, y, 128).cpu().numpy()
    ref = (x.cpu().double().numpy() @ y.cpu().double().numpy())
    f32 = np.where(np.abs(ref) > 3.4028235e38, np.sign(ref) * np.inf, ref)
    same = np.isnan(ref) == np.isnan(got)
    same &= np.isinf(f32) == np.isinf(got)
    same[[60, 90]] |= np.isin(np.arange(100), [9, 10, 11], invert=True)      # (sums of many huge terms pass through infinities in any f32 order; single terms don't)
    assert same.all()
    ok = np.isfinite(f32) & np.isfinite(got)
    scale = np.abs(x.cpu().double().numpy()) @ np.abs(y.cpu().double().numpy())
    assert (np.abs(got - f32)[ok] <= (k * 6e-8 * scale + k * 2.0 ** -149)[ok]).all()


@pytest.mark.parametrize("k", [40, 520])
@pytest.mark.parametrize("small,large", [(1e-35, 1e12), (1e-36, 1e20), (1e-38, 1e25), (1e-40, 1e30), (1e-42, 1e30), (1e-44, 1e30), (1e-25, 1e-15), (1e-28, 1.0), (1e-33, 2e33), (1e-6, 1e31)])
@pytest.mark.parametrize("flip", [False, True])
def test_small_operands_beside_large_ones(mtf, k, small, large, flip):  # noqa: F811
    """Rows of small, ordinary and single small values (whose pieces would lose bits or vanish unscaled) times columns of large, ordinary and small ones: one chain of
    k f32 additions errs by about 2^-24 sqrt(k / 12) of the result, and by half of 2^-149 a term below f32's normal range; twice and more is allowed."""
    import torch
    torch.manual_seed(k)
    dev = {"device": "cuda", "dtype": torch.float64}
    rows, cols = torch.randn(200, k, **dev), torch.randn(k, 100, **dev)
    rows[:60] *= small
    cols[:, :30] *= large
    cols[:, 30:40] *= small
    rows[60:90] = 0.0
    rows[torch.arange(60, 90), torch.arange(60, 90) % k] = small      # one value in a row of zeros
    rows[90:100, 3] = small                                             # ... and beside ordinary ones
    cols[:, 95:] = 0.0
    x, y = rows.float(), cols.float()
    got = product(mtf, y.T.contiguous(), x.T.contiguous(), 128).T if flip else product(mtf, x, y, 128)
    ref, got = x.double() @ y.double(), got.double()
    assert got.isfinite().all()
    for r in (slice(0, 60), slice(60, 90), slice(90, 100), slice(100, 200)):
        for c in (slice(0, 30), slice(30, 40), slice(40, 95), slice(95, 100)):
            e, f = (got - ref)[r, c], ref[r, c]
            assert e.norm() <= 2 ** -24 * k ** 0.5 * f.norm() + k * 2 ** -149 * f.numel() ** 0.5, (r, c)


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (130, 70, 70), (33, 65, 300), (300, 17, 33)])
@pytest.mark.parametrize("order", ["bik,bkj", "bik,bjk", "bki,bkj", "bki,bjk", "ibk,kbj"])
def test_large_operands(mtf, asked, order, m, n, k):  # noqa: F811
    """Values from 2^111 on, in whole rows and columns and alone in one part of K: the second computation, whichever way the operands lie and wherever a
    tile or a run of 32 k ends.  A sum of k products in any order of f32 additions is within k + 1 roundings, 2^-24 of the sum of magnitudes each."""
    import torch
    torch.manual_seed(m)
    size = {"b": 2, "i": m, "j": n, "k": k}
    dev = {"device": "cuda", "dtype": torch.float64}
    x, y = torch.randn(2, m, k, **dev), torch.randn(2, k, n, **dev) * 1e-20
    x[:, : m // 3] *= 2.0 ** 112
    x[1, m - 1, k // 2] = 2.0 ** 120
    y[0, :, n // 2] *= 2.0 ** 60
    a, b = order.split(",")
    tensors = [torch.einsum("%s->%s" % (full, t), v).contiguous().float() for full, t, v in (("bik", a, x), ("bkj", b, y))]
    o = torch.full((2, m, n), float("nan"), device="cuda")
    mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(t, list(names)) for t, names in zip(tensors, (a, b))], mtf.named(o, ["b", "i", "j"]))
    mtf.mtf_device_status()
    ref = torch.einsum("%s,%s->bij" % (a, b), *[t.double() for t in tensors])
    scale = torch.einsum("%s,%s->bij" % (a, b), *[t.double().abs() for t in tensors])
    assert ((o.double() - ref).abs() <= (k + 1) * 2 ** -24 * scale).all()


@pytest.mark.parametrize("order", ["ik,kj", "ki,jk"])
def test_results_out_of_range_cost_what_plain_arithmetic_costs(mtf, order):  # noqa: F811
    """A product of nothing but NaN is computed twice; measured, 4.4 times the time of ordinary values (with each thread computing its own outputs again: 112 times)."""
    import torch
    m, n, k = 1024, 1024, 256
    size = {"i": m, "j": n, "k": k}
    x, y = [torch.randn([size[c] for c in t], device="cuda") for t in order.split(",")]
    o = torch.empty(m, n, device="cuda")
    nan = torch.full_like(x, float("nan"))
    at = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    mtf.mtf_debug_contraction(128, 1)
    for _ in range(2):
        for t, pair in ((x, at[:2]), (nan, at[2:])):
            pair[0].record()
            for _ in range(20):
                mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(t, list(order[:2])), mtf.named(y, list(order[3:]))], mtf.named(o, ["i", "j"]))
            pair[1].record()
    torch.cuda.synchronize()
    assert mtf.mtf_debug_contraction(0, 0)[0] == 128
    assert o.isnan().all()
    assert at[2].elapsed_time(at[3]) <= 9 * at[0].elapsed_time(at[1])


def test_pieces_are_chosen_by_size(mtf):  # noqa: F811
    import torch
    mtf.mtf_debug_contraction(0, 0)
    for m, n, k, ran in ((1024, 1024, 256, 128), (1024, 256, 1024, 128), (8, 256, 64, 128), (256, 64, 16, 64), (1000, 500, 32, 64)):
        x, y, o = torch.randn(m, k, device="cuda"), torch.randn(k, n, device="cuda"), torch.empty(m, n, device="cuda")
        mtf.mtf_einsum(layout(mtf, *ONE), None, [mtf.named(x, ["i", "k"]), mtf.named(y, ["k", "j"])], mtf.named(o, ["i", "j"]))
        assert mtf.mtf_debug_contraction()[0] == ran, (m, n, k)


@pytest.mark.parametrize("tokens,d_in,hidden,d_out", [(1024, 256, 1024, 256), (264, 260, 1028, 260), (1000, 72, 2052, 100), (2048, 40, 1000, 40)])
def test_feed_forward_backward_in_pieces(tokens, d_in, hidden, d_out):
    """dbias comes from the launch of dw, dv and dx run beside the launches before them: every output against 64 bits from what the launch read, the same bits
    from run to run, and launch by launch where dx lies over x."""
    import torch
    import paper_1811_02084_b200 as mtf
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    t = {"x": r(tokens, d_in), "w": r(d_in, hidden) * d_in ** -0.5, "v": r(hidden, d_out) * hidden ** -0.5, "h": r(tokens, hidden).relu(), "dy": r(tokens, d_out)}
    dims = {"x": "td", "w": "df", "v": "fe", "h": "tf", "dy": "te", "dx": "td", "dw": "df", "dbias": "f", "dv": "fe"}
    lay = mtf.mtf_layout(mtf.mtf_mesh_create([("p", 1)]), [])

    def run(over_x):
        o = {"dw": torch.empty(d_in, hidden, device="cuda"), "dbias": torch.empty(hidden, device="cuda"), "dv": torch.empty(hidden, d_out, device="cuda")}
        x = t["x"].clone()
        o["dx"] = x if over_x else torch.empty_like(x)
        for k in ("dw", "dbias", "dv"):
            o[k].fill_(float("nan"))
        n = {k: mtf.named(v, list(dims[k])) for k, v in {**t, **o, "x": x}.items()}
        ws = torch.empty(mtf.mtf_ffn_workspace_bytes(lay, n["x"], n["w"]), dtype=torch.uint8, device="cuda")
        mtf.mtf_ffn_backward(lay, n["x"], n["w"], n["v"], n["h"], n["dy"], n["dx"], n["dw"], n["dbias"], n["dv"], ws)
        mtf.mtf_device_status()
        return o

    first, again, over = run(False), run(False), run(True)
    d = {k: v.double() for k, v in t.items()}
    dhp = (d["dy"] @ d["v"].t()) * (d["h"] > 0)
    ref = {"dv": d["h"].t() @ d["dy"], "dw": d["x"].t() @ dhp, "dx": dhp @ d["w"].t(), "dbias": dhp.sum(0)}
    for k, want in ref.items():
        # (2-norm; sums of up to 2052 terms: the kernel's own error is 1.2e-7 at K = 2048, dhp's rounding 3e-8 more)
        assert (first[k].double() - want).norm() <= 1e-6 * want.norm(), k
        assert torch.equal(first[k], again[k]) and torch.equal(first[k], over[k]), k
