"""The f32 matrix-product kernel against the fp64 oracle: operand orders, sizes around its 64 x 64 tile and 32-deep
k-block, every split of K over a cluster, batch dimensions, exchanged operands and the fused stages."""
import numpy as np
import pytest

import seeded_inputs as si
from helpers import TOL, from_torch, parity_error
from test_gpu_einsum import layout, mtf, run_einsum  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, params=["asked", "chosen"])
def tiled(request, mtf):  # noqa: F811
    """Every test twice: on the tiles, however small the product, and on what the library takes for its size."""
    asked = request.param == "asked"
    mtf.mtf_debug_contraction(*((64, 1) if asked else (0, 0)))
    yield asked
    ran = mtf.mtf_debug_contraction(0, 0)
    assert not asked or ran[0] == 64


# Batches of small products, single rows and columns, short K: one thread per output is many times faster there
SMALL = [(100000, 1, 1, 1), (65536, 2, 2, 8), (4096, 4, 4, 4), (20000, 1, 16, 4), (1000, 8, 8, 8), (1, 1, 200000, 1), (1, 200000, 2, 8), (1, 45, 2, 1)]


@pytest.mark.parametrize("b,m,n,k", SMALL + [(1, 8, 256, 64), (1, 64, 64, 32), (1, 1000, 520, 40), (64, 40, 40, 200)])
def test_small_products_stay_with_one_thread_per_output(mtf, tiled, b, m, n, k):
    import torch
    x, y = torch.randn(b, m, k, device="cuda"), torch.randn(b, k, n, device="cuda")
    out = torch.full((b, m, n), float("nan"), device="cuda")
    mtf.mtf_einsum(layout(mtf, [("all", 1)], []), None, [mtf.named(x, ["b", "i", "k"]), mtf.named(y, ["b", "k", "j"])], mtf.named(out, ["b", "i", "j"]))
    mtf.mtf_device_status()
    assert parity_error(from_torch(out), torch.bmm(x.double(), y.double()).cpu().numpy()) <= TOL["f32"]
    if not tiled:
        assert (mtf.mtf_debug_contraction() == (0, 0)) == ((b, m, n, k) in SMALL)


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (8, 256, 64), (64, 64, 32), (65, 63, 33), (130, 68, 127), (7, 200, 1023), (300, 36, 256), (1000, 520, 40)])
@pytest.mark.parametrize("order", ["ik,kj", "ik,jk", "ki,kj", "ki,jk"])
def test_f32_orders_and_edges(mtf, order, m, n, k):
    size = {"i": m, "j": n, "k": k}
    a, b = [[(c, size[c]) for c in t] for t in order.split(",")]
    for out, dt in ((["i", "j"], "f32"), (["j", "i"], "f32"), (["i", "j"], "bf16")):
        got, ref, info = run_einsum(mtf, layout(mtf, [("all", 1)], []), [a, b], [(c, size[c]) for c in out], "f32", dt)
        assert info["kernel_kind"] == mtf.MTF_KERNEL_SIMT
        assert parity_error(got, ref) <= TOL[dt]


@pytest.mark.parametrize("mesh,rules", [([("all", 1)], []), ([("r", 2), ("c", 2)], [("b", "r"), ("k", "c")])])
def test_f32_batch_dims_and_split_sums(mtf, mesh, rules):
    a, b = [("b", 6), ("i", 40), ("h", 3), ("k", 24)], [("b", 6), ("j", 50), ("h", 3), ("k", 24)]
    got, ref, _ = run_einsum(mtf, layout(mtf, mesh, rules), [a, b], [("b", 6), ("h", 3), ("i", 40), ("j", 50)], "f32")
    assert parity_error(got, ref) <= TOL["f32"]
    a, b = [("b", 6), ("k", 24), ("i", 40)], [("b", 6), ("k", 24), ("j", 50)]
    got, ref, _ = run_einsum(mtf, layout(mtf, mesh, rules), [a, b], [("i", 40), ("j", 50)], "f32")
    assert parity_error(got, ref) <= TOL["f32"]


@pytest.mark.parametrize("m,n,k", [(8, 256, 64), (77, 101, 300), (520, 130, 64)])
@pytest.mark.parametrize("out", [["i", "j"], ["j", "i"]], ids=["in-order", "exchanged"])
def test_f32_stages(mtf, out, m, n, k):
    size = {"i": m, "j": n, "k": k}
    dims = [[(c, size[c]) for c in t] for t in ("ik", "kj")]
    for bias in ("i", "j"):
        ep = {"scale": -0.5, "bias": [(bias, size[bias])], "relu": True, "relu_mask": True, "residual": True}
        got, ref, _ = run_einsum(mtf, layout(mtf, [("all", 1)], []), dims, [(c, size[c]) for c in out], "f32", epilogue=ep)
        assert parity_error(got, ref) <= TOL["f32"]


@pytest.mark.parametrize("m,n,k", [(8, 256, 64), (64, 70, 512), (200, 33, 90), (2000, 64, 64)])
def test_f32_column_sums_and_unaligned_operands(mtf, m, n, k):
    import torch
    x, y = si.normal(3, "x", [m, k], "f32"), si.normal(3, "y", [k, n], "f32")
    dev = []
    for s in (x, y):                                  # operands 4 bytes past a 16-byte boundary
        buf = torch.empty(s.bits.size + 1, device="cuda")
        t = buf[1:].view(*s.bits.shape)
        t.copy_(torch.from_numpy(s.bits.copy()))
        dev.append(t)
    out, col = torch.full((m, n), float("nan"), device="cuda"), torch.full((n,), float("nan"), device="cuda")
    ep = mtf.Epilogue(relu=True, reduce_sum_out=mtf.named(col, ["j"]))
    mtf.mtf_einsum(layout(mtf, [("all", 1)], []), None, [mtf.named(dev[0], ["i", "k"]), mtf.named(dev[1], ["k", "j"])], mtf.named(out, ["i", "j"]), ep)
    mtf.mtf_device_status()
    ref = np.maximum(x.f64 @ y.f64, 0.0)
    assert parity_error(from_torch(out), ref) <= TOL["f32"]
    assert parity_error(from_torch(col), ref.sum(0)) <= TOL["f32"]
