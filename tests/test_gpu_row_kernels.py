"""Row kernels at lengths between their register sizes: layer norm forward and backward at row lengths around multiples of
256 (and beyond the lengths that stay in registers), the cross-entropy's gradient for few and many, short and long rows, and
the table gradient for row lengths with and without whole 16-byte pieces; against fp64 arithmetic on the same inputs."""
import numpy as np
import pytest

import seeded_inputs as si
from helpers import TOL, from_torch, parity_error, to_torch
from test_gpu_einsum import layout, mtf  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 248, 264, 512, 520, 776, 1016, 1032, 1288, 1544, 1800, 2040, 2056])
@pytest.mark.parametrize("rows", [1, 77, 3001])
@pytest.mark.parametrize("scratch", [False, True])
def test_layernorm_lengths(mtf, n, rows, scratch):
    import torch
    lay = layout(mtf, [("all", 1)], [])
    x, dy, res = (si.normal(4, k, [rows, n], "bf16") for k in ("x", "dy", "res"))
    g, b = si.normal(4, "g", [n], "f32"), si.normal(4, "b", [n], "f32")
    tx, tdy, tres, tg, tb = (to_torch(s) for s in (x, dy, res, g, b))
    y, dx = torch.full((rows, n), float("nan"), dtype=torch.bfloat16, device="cuda"), torch.full((rows, n), float("nan"), dtype=torch.bfloat16, device="cuda")
    stats, dg, db = torch.empty(rows, 2, device="cuda"), torch.full((n,), float("nan"), device="cuda"), torch.full((n,), float("nan"), device="cuda")
    N = mtf.named
    mtf.mtf_layernorm_forward(lay, N(tx, ["t", "c"]), N(tg, ["c"]), N(tb, ["c"]), 1e-6, N(y, ["t", "c"]), N(stats, ["t", "two"]))
    size = mtf.mtf_layernorm_workspace_bytes(n)
    assert (size > 0) == (n <= 2048)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda") if scratch and size else None
    runs = []
    for _ in range(4 if ws is not None else 1):
        dg.fill_(float("nan"))
        db.fill_(float("nan"))
        mtf.mtf_layernorm_backward(lay, N(tdy, ["t", "c"]), N(tx, ["t", "c"]), N(stats, ["t", "two"]), N(tg, ["c"]), N(tres, ["t", "c"]), N(dx, ["t", "c"]), N(dg, ["c"]),
                                   N(db, ["c"]), ws)
        runs.append((dg.clone(), db.clone()))
    mtf.mtf_device_status()
    assert all(torch.equal(a, b) for r in runs[1:] for a, b in zip(runs[0], r))        # (with the scratch that the query asks for)
    mu = x.f64.mean(1, keepdims=True)
    rstd = 1 / np.sqrt(((x.f64 - mu) ** 2).mean(1, keepdims=True) + 1e-6)
    xh = (x.f64 - mu) * rstd
    assert parity_error(from_torch(y), g.f64 * xh + b.f64) <= TOL["bf16"]
    assert parity_error(from_torch(stats), np.concatenate([mu, rstd], 1)) <= TOL["f32"]
    gg = dy.f64 * g.f64
    assert parity_error(from_torch(dx), rstd * (gg - gg.mean(1, keepdims=True) - xh * (gg * xh).mean(1, keepdims=True)) + res.f64) <= TOL["bf16"]
    assert parity_error(from_torch(dg), (dy.f64 * xh).sum(0)) <= TOL["f32"]
    assert parity_error(from_torch(db), dy.f64.sum(0)) <= TOL["f32"]


@pytest.mark.parametrize("vocab", [8, 264, 2040, 2048, 5000, 9000, 50000])
@pytest.mark.parametrize("rows", [1, 9, 1500])
def test_cross_entropy_gradient(mtf, vocab, rows):
    import torch
    lay = layout(mtf, [("all", 1)], [])
    z, w = si.normal(5, "z", [rows, vocab], "bf16", 2.0), si.normal(5, "w", [rows], "f32")
    tz, tw = to_torch(z), to_torch(w)
    target = torch.from_numpy(np.random.RandomState(1).randint(0, vocab, rows).astype(np.int32)).cuda()
    lse, loss = torch.empty(rows, device="cuda"), torch.empty(rows, device="cuda")
    N = mtf.named
    mtf.mtf_softmax_xent_forward(lay, N(tz, ["t", "v"]), target, N(lse, ["t"]), N(loss, ["t"]))
    mtf.mtf_softmax_xent_backward(lay, N(tz, ["t", "v"]), target, N(lse, ["t"]), N(tw, ["t"]))
    mtf.mtf_device_status()
    ref = np.exp(z.f64 - np.log(np.exp(z.f64).sum(1, keepdims=True)))
    ref[np.arange(rows), target.cpu().numpy()] -= 1
    assert parity_error(from_torch(tz), ref * w.f64[:, None]) <= TOL["bf16"]


@pytest.mark.parametrize("d", [3, 6, 8, 260])
@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_table_gradient(mtf, d, dtype):
    import torch
    dx = si.normal(6, "dx", [700, d], dtype)
    ids = np.random.RandomState(2).randint(0, 50, 700).astype(np.int32)
    out = torch.full((50, d), float("nan"), device="cuda")
    mtf.mtf_embedding_backward(layout(mtf, [("all", 1)], []), torch.from_numpy(ids).cuda(), mtf.named(to_torch(dx), ["t", "c"]), mtf.named(out, ["v", "c"]))
    mtf.mtf_device_status()
    ref = np.zeros((50, d))
    np.add.at(ref, ids, dx.f64)
    assert parity_error(from_torch(out), ref) <= TOL["f32"]
