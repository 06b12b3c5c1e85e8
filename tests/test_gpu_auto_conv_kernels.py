"""The kernels a training step chooses by itself (impl "auto") at the edges of
their rules: one row, one less and one more than a 128-row tile, more items
than CTAs, every channel count the rule names, one and several k-steps, one and
several column units, raw fp32 inputs.  Each launch is held to the oracle and
the bounds of test_gpu_conv_kernels; test_conv_choice_cpu asserts that these are
the cases the rules take."""
import pytest

import test_gpu_conv_kernels as K

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2103_08802_gb300 import build
    build.build()


def _pw(batch, h, w, c, k, **kw):
    return dict(batch=batch, h=h, w=w, c=c, k=k, ksize=1, stride=1, **kw)


PW = {
    "m1": _pw(1, 1, 1, 16, 64, bn=True),
    "m127": _pw(1, 127, 1, 64, 16, bn=True),
    "m128": _pw(2, 8, 8, 32, 128, bn=True),
    "m129": _pw(3, 43, 1, 16, 16, bn=True, relu=False),
    "m31": _pw(1, 31, 1, 32, 32, bn=False),
    "c128_k32": _pw(2, 15, 15, 128, 32, bn=True),
    "c256_k64": _pw(2, 9, 15, 256, 64, bn=True),
    "c64_k256": _pw(3, 9, 15, 64, 256, bn=True),
    "c64_k192": _pw(1, 20, 20, 64, 192, bn=True),
    "c64_k64_fp32x": _pw(2, 15, 15, 64, 64, bn=True, x_fp32=True),
    "many_k64": _pw(6, 100, 100, 16, 64, bn=True),     # 469 m-tiles: whole rows of units an item
    "many_k256": _pw(5, 100, 101, 32, 256, bn=True),   # 395 m-tiles, four units each
    "many_k16": _pw(5, 100, 101, 128, 16, bn=True),
    "expand": [_pw(2, 16, 16, 16, 64, bn=True), _pw(2, 9, 9, 64, 256, bn=True)],
    "reduce": [_pw(2, 16, 16, 64, 16, bn=True), _pw(2, 9, 9, 256, 64, bn=False)],
}
# epilogues: 0 bf16 y, 2 bf16 y + bf16 residual; a group's second instance takes the next of three, so 2 gives
# both (1, fp32 y and residual, is not these kernels')
CASES = [(n, kind) for n in PW for kind in ([2] if isinstance(PW[n], list) else [0, 2])]


def _install(monkeypatch, name, spec):
    if isinstance(spec, list):
        monkeypatch.setitem(K.GROUPS, name, spec)
    else:
        monkeypatch.setitem(K.CASES, name, spec)


@pytest.mark.parametrize("base,kind", CASES)
def test_pointwise_forward(monkeypatch, base, kind):
    _install(monkeypatch, base, PW[base])
    K.check_forward(base, "auto", kind)


@pytest.mark.parametrize("base", list(PW))
def test_pointwise_data_gradient(monkeypatch, base):
    _install(monkeypatch, base, PW[base])
    K.test_conv_data_gradient(base, "auto")


def test_nonfinite_residual_stays_in_its_element():
    """An infinite residual element makes that output infinite and no other."""
    import torch
    from paper_2103_08802_gb300 import pnn
    torch.manual_seed(3)
    d = dict(batch=1, h=16, w=16, c=16, k=64, ksize=1, stride=1)
    d["x"] = torch.randn(1, 16, 16, 16, device="cuda").bfloat16()
    d["wt"] = torch.randn(64, 1, 1, 16, device="cuda").bfloat16()
    d["y"] = torch.empty(1, 16, 16, 64, dtype=torch.bfloat16, device="cuda")
    d["res"] = torch.randn(1, 16, 16, 64, device="cuda").bfloat16()
    d["res"][0, 3, 5, 7] = float("inf")
    pnn.conv_run("forward", [d])
    bad = ~torch.isfinite(d["y"].float())
    assert bad.sum().item() == 1 and bad[0, 3, 5, 7].item()


def _wg(batch, h, w, c, k, ks, **kw):
    return dict(batch=batch, h=h, w=w, c=c, k=k, ksize=ks, stride=1, **kw)


WG = {
    "one_pixel": _wg(1, 1, 1, 16, 64, 1, bn=True),
    "m127": _wg(1, 127, 1, 64, 16, 1, bn=True),
    "m129": _wg(3, 43, 1, 32, 32, 1, bn=True, relu=False),
    "many": _wg(5, 100, 101, 16, 64, 1, bn=True),        # several k-steps a split, a ragged last one
    "k256": _wg(3, 20, 20, 64, 256, 1, bn=True),         # two halves of the M side, gradient on it
    "c256": _wg(3, 20, 20, 256, 64, 1, bn=True),         # ... activation on it
    "c256_fp32x": _wg(2, 15, 15, 256, 16, 1, bn=True, x_fp32=True),
    "c128_raw": _wg(2, 15, 15, 128, 32, 1, bn=False),
    "group_1x1": [_wg(2, 16, 16, 64, 16, 1, bn=True), _wg(2, 8, 8, 128, 32, 1, bn=True),
                  _wg(2, 4, 4, 256, 64, 1, bn=True)],
    "w32": _wg(3, 32, 32, 16, 16, 3, bn=True),
    "w32_h6": _wg(2, 6, 32, 16, 32, 3, bn=True),         # k-steps of three rows
    "w16_h5": _wg(3, 5, 16, 32, 16, 3, bn=True),         # one k-step an image
    "w8": _wg(3, 8, 8, 64, 64, 3, bn=True),              # two channel halves, row-strided pixel groups
    "w8_h16_k128": _wg(2, 16, 8, 32, 128, 3, bn=False),
    "w16_fp32x": _wg(2, 16, 16, 64, 16, 3, bn=True, x_fp32=True, relu=False),
    "w16_c128_k128": _wg(2, 16, 16, 128, 128, 3, bn=True),   # four blocks of input channels
    "w8_c96_k256": _wg(3, 8, 8, 96, 256, 3, bn=True, relu=False),  # three by two blocks
    "small4x4": _wg(9, 4, 4, 64, 128, 3, bn=True),           # whole images, a ragged last k-step
    "small2x2": _wg(70, 2, 2, 32, 256, 3, bn=True),
    "small1x1": _wg(130, 1, 1, 16, 32, 3, bn=True),
    "small2x8_fp32x": _wg(5, 2, 8, 32, 16, 3, bn=True, x_fp32=True),
    "group_kinds": [_wg(20, 4, 4, 64, 64, 3, bn=True), _wg(2, 16, 16, 32, 128, 3, bn=True)],
    "group_3x3": [_wg(4, 32, 32, 16, 16, 3, bn=True), _wg(2, 16, 16, 32, 32, 3, bn=True),
                  _wg(2, 8, 8, 64, 64, 3, bn=True)],
}


@pytest.mark.parametrize("base", list(WG))
def test_weight_gradient(monkeypatch, base):
    _install(monkeypatch, base, WG[base])
    K.test_conv_weight_gradient(base, "auto")


C3 = {
    "patch": _wg(1, 16, 8, 16, 16, 3, bn=True),
    "patches": _wg(3, 32, 32, 16, 16, 3, bn=True),
    "p48x24": _wg(2, 48, 24, 32, 16, 3, bn=True, relu=False),
    "p16x40_n64": _wg(2, 16, 40, 16, 64, 3, bn=False),
    "p16_c64": _wg(2, 16, 16, 64, 64, 3, bn=True),
    "p16_c64_fp32x": _wg(2, 16, 16, 64, 32, 3, bn=True, x_fp32=True),
    "whole1": _wg(1, 8, 8, 16, 32, 3, bn=True),           # half a tile
    "whole5": _wg(5, 8, 8, 64, 64, 3, bn=True),
    "many": _wg(20, 64, 32, 16, 16, 3, bn=True),          # more tiles than CTAs
    "p16_c128_n192": _wg(2, 16, 16, 128, 192, 3, bn=True),   # eight k-steps, three column blocks
    "whole_c192_n128": _wg(3, 8, 8, 192, 128, 3, bn=True, relu=False),
    "small4x4": _wg(9, 4, 4, 64, 128, 3, bn=True),        # a full tile and one image
    "small2x2": _wg(33, 2, 2, 128, 64, 3, bn=True),
    "small1x1": _wg(129, 1, 1, 16, 32, 3, bn=True),
    "small2x8_fp32x": _wg(5, 2, 8, 32, 16, 3, bn=True, x_fp32=True),
    "small_kinds": [_wg(20, 4, 4, 64, 64, 3, bn=True), _wg(2, 16, 16, 32, 128, 3, bn=True)],
    "small_whole": [_wg(3, 8, 8, 64, 128, 3, bn=True), _wg(40, 2, 2, 128, 64, 3, bn=False)],
    "stages": [_wg(2, 32, 32, 16, 16, 3, bn=True), _wg(3, 8, 8, 64, 64, 3, bn=True)],
    "stages_reversed": [_wg(3, 8, 8, 64, 64, 3, bn=True), _wg(2, 16, 16, 32, 32, 3, bn=True)],
}


@pytest.mark.parametrize("base,kind", [(n, kind) for n in C3 for kind in ([2] if isinstance(C3[n], list) else [0, 2])])
def test_3x3_forward(monkeypatch, base, kind):
    _install(monkeypatch, base, C3[base])
    K.check_forward(base, "auto", kind)


@pytest.mark.parametrize("base", list(C3))
def test_3x3_data_gradient(monkeypatch, base):
    _install(monkeypatch, base, C3[base])
    K.test_conv_data_gradient(base, "auto")


@pytest.mark.parametrize("mode,c,k,ks", [("forward", 16, 64, 1), ("forward", 16, 16, 3), ("wgrad", 16, 64, 1),
                                         ("wgrad", 16, 16, 3)])
def test_per_channel_values_at_odd_offsets(mode, c, k, ks):
    """BN scale and shift may be slices at any float offset: such a call keeps the
    kernels that read them one at a time, whose result is that of impl "tma"."""
    import torch
    from paper_2103_08802_gb300 import pnn
    torch.manual_seed(5)
    b, h = 3, 32
    base = dict(batch=b, h=h, w=h, c=c, k=k, ksize=ks, stride=1, relu=1)
    base["x"] = torch.randn(b, h, h, c, device="cuda").bfloat16()
    base["wt"] = torch.randn(k, ks, ks, c, device="cuda").bfloat16()
    base["dy"] = torch.randn(b, h, h, k, device="cuda")
    buf = torch.rand(2, c + 1, device="cuda") + 0.5
    results = []
    for impl, odd in (("tma", False), ("auto", True)):
        d = dict(base)
        for i, name in enumerate(("bn_scale", "bn_shift")):
            t = torch.empty(c + 1, device="cuda")[1:] if odd else torch.empty(c, device="cuda")
            t.copy_(buf[i, 1:])
            assert t.data_ptr() % 8 == (4 if odd else 0)
            d[name] = t
        d["y"] = torch.zeros(b, h, h, k, device="cuda", dtype=torch.bfloat16)
        d["dw"] = torch.zeros(k, ks, ks, c, device="cuda")
        pnn.conv_run(mode, [d], impl=impl)
        results.append(d["y"] if mode == "forward" else d["dw"])
    assert results[0].abs().max() > 0 and torch.equal(results[0], results[1])


@pytest.mark.parametrize("ks,c,k", [(1, 64, 16), (3, 16, 16)])
@pytest.mark.parametrize("odd", ["bn_scale", "bn_shift", "bn_mean", "bn_rstd"])
def test_data_gradient_sums_with_values_at_odd_offsets(odd, ks, c, k):
    """Each of the BN values of a data gradient's sums in turn at an odd float offset: dx is that of impl "tma",
    the sums (of another kernel, in another order) within the bound of any order of the same fp32 terms."""
    import torch
    from paper_2103_08802_gb300 import pnn
    torch.manual_seed(6)
    b, h = 3, 32
    rows = b * h * h
    base = dict(batch=b, h=h, w=h, c=c, k=k, ksize=ks, stride=1, relu=1)
    base["x"] = torch.randn(b, h, h, c, device="cuda").bfloat16()
    base["wt"] = torch.randn(k, ks, ks, c, device="cuda").bfloat16()
    base["dy"] = torch.randn(b, h, h, k, device="cuda")
    values = {n: torch.rand(c, device="cuda") + 0.5 for n in ("bn_scale", "bn_shift", "bn_mean", "bn_rstd")}
    dx = []
    for impl, shifted in (("tma", None), ("auto", odd)):
        d = dict(base, dx=torch.zeros(b, h, h, c, device="cuda"))
        for n, v in values.items():
            d[n] = torch.empty(c + 1, device="cuda")[1:] if n == shifted else torch.empty(c, device="cuda")
            d[n].copy_(v)
            assert d[n].data_ptr() % 8 == (4 if n == shifted else 0)
        d["dgamma"], d["dbeta"] = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
        pnn.conv_run("dgrad", [d], impl=impl)
        dx.append(d["dx"])
        x = base["x"].view(-1, c)
        pre = (values["bn_scale"].double() * x.double() + values["bn_shift"].double()).float()
        g = torch.where(pre > 0, d["dx"].view(-1, c), torch.zeros((), device="cuda")).double()
        xh = ((x.float() - values["bn_mean"]) * values["bn_rstd"]).double()
        for got, term in ((d["dbeta"], g), (d["dgamma"], g * xh)):
            assert ((got.double() - term.sum(0)).abs() <= rows * K.U * term.abs().sum(0)).all()
    assert torch.equal(dx[0], dx[1])


def _flat(rows, c, k):
    return dict(batch=1, h=rows, w=1, c=c, k=k, ksize=1)


# layers whose last tile leaves whole warps without rows (rows % 128 in 1 .. 96), after full tiles of the
# same warps: 64 columns (two staged blocks a unit), and 16 or 32 (one) in groups of more tiles than CTAs,
# where a CTA goes from such a tile to another layer's
RAGGED = {
    "dgrad_1x1_c64": ("dgrad", "auto", [_flat(60000, 64, 16)]),
    "dgrad_1x1_c256": ("dgrad", "auto", [_flat(20000 + 33, 256, 64)]),
    "dgrad_1x1_group": ("dgrad", "auto", [_flat(257, 16 * (1 + i % 2), 16) for i in range(150)]),
    "dgrad_3x3_c64": ("dgrad", "auto", [dict(batch=401, h=8, w=8, c=64, k=16, ksize=3)]),
    "dgrad_3x3_group": ("dgrad", "auto", [dict(batch=5, h=8, w=8, c=16 * (1 + i % 2), k=16, ksize=3) for i in range(120)]),
    "dgrad_3x3_small": ("dgrad", "auto", [dict(batch=8 * 40 + 1, h=4, w=4, c=128, k=64, ksize=3)]),
    "dgrad_tma": ("dgrad", "tma", [_flat(60000, 64, 64)]),
    "dgrad_tma_group": ("dgrad", "tma", [_flat(257, 16, 64) for i in range(150)]),
    "dgrad_tma_tap": ("dgrad", "tma_tap", [dict(batch=401, h=8, w=8, c=64, k=64, ksize=3)]),
    "forward_1x1_k64": ("forward", "auto", [_flat(60000, 16, 64)]),
    "forward_tma": ("forward", "tma", [_flat(60000, 64, 128)]),
    "forward_tma_group": ("forward", "tma", [_flat(257, 64, 64) for i in range(150)]),
}


@pytest.mark.parametrize("name,accumulate", [(n, a) for n in RAGGED for a in ([0, 1] if n.startswith("dgrad") else [0])])
def test_staged_tiles_next_to_empty_rows(name, accumulate):
    """Small whole numbers, so every sum is exact; no BN sums between a staged tile and the next."""
    import torch
    import torch.nn.functional as F
    from paper_2103_08802_gb300 import pnn
    mode, impl, geo = RAGGED[name]
    torch.manual_seed(7)
    ints = lambda *s: torch.randint(-1, 2, s, device="cuda").float()  # noqa: E731
    insts, want = [], []
    for g in geo:
        d = dict(g, stride=1)
        b, h, w, c, k, ks = (d[n] for n in ("batch", "h", "w", "c", "k", "ksize"))
        wt, src = ints(k, ks, ks, c), ints(b, h, w, c if mode == "forward" else k)
        d["wt"] = wt.bfloat16()
        kern = wt.double().permute(0, 3, 1, 2)
        x = src.double().permute(0, 3, 1, 2)
        if mode == "forward":
            d["x"], d["y"] = src.bfloat16(), torch.empty(b, h, w, k, device="cuda", dtype=torch.bfloat16)
            want.append(F.conv2d(x, kern, padding=ks // 2).permute(0, 2, 3, 1))
        else:
            d["dy"], d["dx"], d["accumulate"] = src, torch.empty(b, h, w, c, device="cuda"), accumulate
            want.append(F.conv_transpose2d(x, kern, padding=ks // 2).permute(0, 2, 3, 1))
        insts.append(d)
    for _ in range(8):
        for d in insts:
            d["y" if mode == "forward" else "dx"].fill_(3.0)
        pnn.conv_run(mode, insts, impl=impl)
        for d, e in zip(insts, want):
            got = d["y" if mode == "forward" else "dx"].double()
            assert torch.equal(got, e + 3.0 if accumulate else e)


def test_trace_names_the_kernels_of_a_network():
    import torch
    import workloads as W
    from paper_2103_08802_gb300 import pnn
    desc = W.parareal_resnet1001(n_seg=2, batch=16, per_stage=2)
    net = pnn.ParaNet(desc, seed=1, lr=0.002)
    x, labels = W.make_batch(desc, seed=3)
    net.profile(True)
    net.forward(torch.from_numpy(x).cuda(), torch.from_numpy(labels).cuda())
    net.backward()
    trace = net.profile_trace()
    net.close()
    tc = ("conv_fwd_tc", "conv_dgrad_tc", "conv_wgrad_tc")
    assert all((r["kernel"] is not None) == (r["kind"] in tc) for r in trace)
    # 1x1 and 3x3 layers, the stride-2 ones, and the last convolution of a subnetwork (a correction addend)
    assert {r["kernel"] for r in trace} >= {"k_pw_fwd", "k_pw_fwd_w", "k_pw_dgrad", "k_c3_fwd<false>", "k_c3_dgrad<false>",
                                            "k_wg_pw", "k_wg_3x3<false>", "k_conv_fwd_tc", "k_conv_dgrad_tc"}
    assert any(r["kernel"].startswith("k_conv_fwd_tma") for r in trace if r["kind"] == "conv_fwd_tc")
