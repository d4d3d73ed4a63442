"""The f32 feed-forward block on a few tokens (one launch a direction) against 64-bit arithmetic: sizes that eight blocks, four rows or eight terms do not
divide, each output from the values the launch read, and the calls that stay with one launch per einsum."""
import pytest

from test_gpu_einsum import layout, mtf  # noqa: F401

pytestmark = pytest.mark.gpu


def block(T, D, F, E, bias=True, seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = {k: torch.randn(*s, generator=g, device="cuda") * c for k, s, c in
         (("x", (T, D), 1.0), ("w", (D, F), D ** -0.5), ("bias", (F,), 0.1), ("v", (F, E), F ** -0.5), ("dy", (T, E), 1.0))}
    for k, s in (("h", (T, F)), ("y", (T, E)), ("dx", (T, D)), ("dw", (D, F)), ("dbias", (F,)), ("dv", (F, E))):
        t[k] = torch.full(s, float("nan"), device="cuda")
    if not bias:
        t["bias"] = t["dbias"] = None
    return t


DIMS = {"x": ["t", "d"], "w": ["d", "f"], "bias": ["f"], "v": ["f", "e"], "dy": ["t", "e"], "h": ["t", "f"], "y": ["t", "e"], "dx": ["t", "d"], "dw": ["d", "f"],
        "dbias": ["f"], "dv": ["f", "e"]}


def run(mtf, lay, t, dims=DIMS):  # noqa: F811
    import torch
    n = {k: None if v is None else mtf.named(v, dims[k]) for k, v in t.items()}
    ws = torch.empty(mtf.mtf_ffn_workspace_bytes(lay, n["x"], n["w"]), dtype=torch.uint8, device="cuda")
    before = mtf.mtf_launch_count()
    mtf.mtf_ffn_forward(lay, n["x"], n["w"], n["bias"], n["v"], n["h"], n["y"], ws)
    mtf.mtf_ffn_backward(lay, n["x"], n["w"], n["v"], n["h"], n["dy"], n["dx"], n["dw"], n["dbias"], n["dv"], ws)
    mtf.mtf_device_status()
    return mtf.mtf_launch_count() - before


def check(t, dy=None):
    """2-norm errors.  A result is rounded once (2^-24); what it is made of were sums of eight terms in f32 (at most seven roundings of 2^-24 of the terms'
    sizes, which cancel at most sqrt(8) to 1 in the 2-norm of a normal sum), and dhp was rounded before dw, dx and dbias: below 1e-6 in all."""
    d = {k: v.double() for k, v in t.items() if v is not None}
    dy = d["dy"] if dy is None else dy.double()
    dhp = (dy @ d["v"].t()) * (d["h"] > 0)
    ref = {"h": (d["x"] @ d["w"] + d.get("bias", 0.0)).relu(), "y": d["h"] @ d["v"], "dv": d["h"].t() @ dy, "dw": d["x"].t() @ dhp, "dx": dhp @ d["w"].t(), "dbias": dhp.sum(0)}
    for k, r in ref.items():
        if k in d:
            assert (d[k] - r).norm() <= 1e-6 * r.norm(), k


@pytest.mark.parametrize("T,D,F,E", [(1, 1, 1, 1), (8, 64, 256, 64), (5, 7, 9, 3), (3, 40, 72, 24), (17, 33, 130, 65), (2, 512, 8, 9), (130, 5, 20, 12), (33, 64, 100, 8)])
@pytest.mark.parametrize("bias", [True, False])
def test_edges(mtf, T, D, F, E, bias):  # noqa: F811
    import torch
    t = block(T, D, F, E, bias)
    assert run(mtf, layout(mtf, [("all", 1)], []), t) == 2
    check(t)
    again = block(T, D, F, E, bias)
    run(mtf, layout(mtf, [("all", 1)], []), again)
    assert all(v is None or torch.equal(v, again[k]) for k, v in t.items())


def test_layouts_and_token_dims(mtf):  # noqa: F811
    import torch
    flat = block(12, 40, 72, 40)
    run(mtf, layout(mtf, [("all", 1)], []), flat)
    t = {k: v.clone() for k, v in block(12, 40, 72, 40).items()}
    for k in ("x", "dy", "h", "y", "dx"):
        t[k] = t[k].view(4, 3, -1)
    dims = {k: (["b", "l"] + v[1:] if v[0] == "t" else v) for k, v in DIMS.items()}
    assert run(mtf, layout(mtf, [("r", 2), ("c", 4)], [("b", "r"), ("f", "c")]), t, dims) == 2
    assert all(torch.equal(t[k].reshape(flat[k].shape), flat[k]) for k in flat)
    with pytest.raises(mtf.MtfError):               # what no layout allows is still refused
        run(mtf, layout(mtf, [("r", 5)], [("f", "r")]), block(12, 40, 72, 40))


def test_outputs_over_operands_go_launch_by_launch(mtf):  # noqa: F811
    t = block(8, 64, 256, 64)
    dy = t["dy"].clone()
    t["dx"] = t["dy"]                               # dx over dy: every launch that reads dy comes before the one that writes dx
    assert run(mtf, layout(mtf, [("all", 1)], []), t) > 2
    check(t, dy)


def test_non_finite_values_stay_in_their_rows(mtf):  # noqa: F811
    import torch
    t, clean = block(9, 40, 72, 40), block(9, 40, 72, 40)
    t["dy"][4, 3] = float("nan")
    t["x"][6, 1] = float("inf")
    lay = layout(mtf, [("all", 1)], [])
    run(mtf, lay, t)
    run(mtf, lay, clean)
    rows = torch.tensor([i for i in range(9) if i not in (4, 6)], device="cuda")
    assert torch.equal(t["y"][rows], clean["y"][rows]) and torch.equal(t["dx"][rows], clean["dx"][rows])
    assert t["dx"][4].isnan().all() and t["dv"].isnan()[:, 3].any() and t["h"][6].isinf().any()


@pytest.mark.parametrize("T,D,F,E", [(8, 64, 256, 64), (64, 40, 72, 40), (5, 200, 300, 100), (24, 64, 128, 64)])
def test_sums_are_exact_to_a_few_roundings(mtf, T, D, F, E):  # noqa: F811
    """A rounding of a value costs 0.41 x 2^-24 of it in the root mean square.  A sum of normal terms with chains of four in f32, f64 between them and one
    rounding at the end has the variance of (1 + 2 + 3 + 4) / 4 + 1 = 3.5 roundings of the result: 0.77 x 2^-24.  Chains of eight would have 5.5: 0.96."""
    num = {"h": 0.0, "y": 0.0, "dv": 0.0}
    den = dict(num)
    for seed in range(8):
        t = block(T, D, F, E, bias=False, seed=seed)
        run(mtf, layout(mtf, [("all", 1)], []), t)
        d = {k: v.double() for k, v in t.items() if v is not None}
        for k, ref in (("h", (d["x"] @ d["w"]).relu()), ("y", d["h"] @ d["v"]), ("dv", d["h"].t() @ d["dy"])):
            num[k] += float((d[k] - ref).norm()) ** 2
            den[k] += float(ref.norm()) ** 2
    for k in num:
        assert (num[k] / den[k]) ** 0.5 <= 0.87 * 2.0 ** -24, (k, (num[k] / den[k]) ** 0.5 * 2.0 ** 24)
