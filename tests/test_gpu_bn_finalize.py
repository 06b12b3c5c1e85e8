"""The BN finalisation kernels at the edges of their tile loop: one partial
tile, one less and one more than the tile lanes of a CTA, more than one round
of loads, a ragged last tile, channels that do not fill the CTA's group.

The statistics are compared with float64 ones of the values the kernel stored.
Bounds: a tile's mean and M2 are fp32 sums of 128 terms (at most 32 in a row,
merged in fours), so each is within 40 u of its sum of absolute terms; the
finalisation forms d = mean_t - mean_0, n d and M2 + n d^2 in fp32, one rounding
each (the forward's terms have 24 bits), and adds them to about 48 bits, the
backward's sums to more than 53.  64 u covers the forward's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U = 2.0 ** -24

ROWS = [1, 100, 63 * 128, 64 * 128, 64 * 128 + 1, 1024 * 128 + 5, 1025 * 128]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2103_08802_gb300 import build
    build.build()


def _shape(rows):
    """batch, h, w with batch * h * w = rows"""
    for h in range(int(rows ** 0.5), 0, -1):
        if rows % h == 0:
            return 1, h, rows // h


@pytest.mark.parametrize("k", [8, 24, 64])
@pytest.mark.parametrize("rows", ROWS)
def test_forward_statistics(rows, k):
    import torch
    from paper_2103_08802_gb300 import pnn
    torch.manual_seed(rows + k)
    b, h, w = _shape(rows)
    d = dict(batch=b, h=h, w=w, c=16, k=k, ksize=1, stride=1)
    d["x"] = (torch.randn(b, h, w, 16, device="cuda") + 0.5).bfloat16()
    d["wt"] = torch.randn(k, 1, 1, 16, device="cuda").bfloat16()
    d["y"] = torch.empty(b, h, w, k, dtype=torch.bfloat16, device="cuda")
    d["y_mean"], d["y_rstd"] = torch.empty(k, device="cuda"), torch.empty(k, device="cuda")
    pnn.conv_run("forward", [d])
    y = d["y"].view(-1, k).double()
    mean, var = y.mean(0), y.var(0, unbiased=False)
    err = (d["y_mean"].double() - mean).abs() / y.abs().mean(0)
    assert err.max().item() <= 64 * U
    rel = (d["y_rstd"].double() * (var + 1e-5).sqrt() - 1).abs()
    assert rel.max().item() <= 64 * U


@pytest.mark.parametrize("c", [8, 16, 72])
@pytest.mark.parametrize("rows", ROWS)
def test_backward_sums(rows, c):
    import torch
    from paper_2103_08802_gb300 import pnn
    torch.manual_seed(rows + c)
    b, h, w = _shape(rows)
    d = dict(batch=b, h=h, w=w, c=c, k=16, ksize=1, stride=1, relu=1)
    d["x"] = torch.randn(b, h, w, c, device="cuda").bfloat16()
    d["wt"] = torch.randn(16, 1, 1, c, device="cuda").bfloat16()
    d["bn_scale"], d["bn_shift"] = torch.rand(c, device="cuda") + 0.5, 0.3 * torch.randn(c, device="cuda")
    d["bn_mean"], d["bn_rstd"] = 0.1 * torch.randn(c, device="cuda"), torch.rand(c, device="cuda") + 0.5
    d["dy"] = torch.randn(b, h, w, 16, device="cuda")
    d["dx"] = torch.empty(b, h, w, c, device="cuda")
    d["dgamma"], d["dbeta"] = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
    pnn.conv_run("dgrad", [d])
    # the mask and xhat as the kernel forms them, in fp32; their products and sums in fp64
    x = d["x"].view(-1, c).float()
    pre = (d["bn_scale"].double() * x.double() + d["bn_shift"].double()).float()  # one rounding: a fused multiply-add
    g = torch.where(pre > 0, d["dx"].view(-1, c), torch.zeros((), device="cuda")).double()
    xh = ((x - d["bn_mean"]) * d["bn_rstd"]).double()
    # the largest tile has 4096 rows (c = 8): at most 128 terms in a row a thread, then a tree
    for got, term in ((d["dbeta"], g), (d["dgamma"], g * xh)):
        err = (got.double() - term.sum(0)).abs()
        assert (err <= 160 * U * term.abs().sum(0) + 1e-30).all(), float((err / term.abs().sum(0)).max())


def test_backward_sums_keep_fp64_bits():
    """Partials of one column that need 53 bits together and cancel to the last of them: the tiles that one
    thread of the finalisation adds (128 apart) hold 2^30, 8, 2^-22, -8, -2^30."""
    import torch
    from paper_2103_08802_gb300 import pnn
    rows, c = 513 * 128, 16
    d = dict(batch=1, h=rows, w=1, c=c, k=c, ksize=1, stride=1, relu=0)
    d["x"] = torch.ones(1, rows, 1, c, device="cuda").bfloat16()
    d["wt"] = torch.eye(c, device="cuda").view(c, 1, 1, c).bfloat16()
    for n, v in (("bn_scale", 1.0), ("bn_shift", 0.0), ("bn_mean", 0.0), ("bn_rstd", 1.0)):
        d[n] = torch.full((c,), v, device="cuda")
    d["dy"] = torch.zeros(1, rows, 1, c, device="cuda")
    for i, v in enumerate((2.0 ** 30, 8.0, 2.0 ** -22, -8.0, -2.0 ** 30)):
        d["dy"][0, i * 128 * 128, 0, 3] = v
    d["dx"] = torch.empty(1, rows, 1, c, device="cuda")
    d["dgamma"], d["dbeta"] = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
    pnn.conv_run("dgrad", [d])
    want = torch.zeros(c, device="cuda")
    want[3] = 2.0 ** -22
    assert torch.equal(d["dbeta"], want) and torch.equal(d["dgamma"], want)
