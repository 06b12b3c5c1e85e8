"""The CUDA-core kernels (convolutions, split reduction, elementwise sums,
pooling, head) at channel counts and sizes where their tiles end: small untorn
and torn networks in fp32 check mode against the oracle, within the 1e-4 of
that mode.  Channel counts on both sides of the tile widths (16, 32, 64), inputs
of 1, 3 and 7 channels (few-channel kernels: at most 32 taps x channels),
strides, odd images, pools whose channel count is no multiple of four, heads
with one and with several groups of K."""
import pytest

import workloads as W
from parity import compare, inputs, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2103_08802_gb300 import build
    build.build()


def _net(name, batch, in_c, h, w, stem, body, classes=7, hidden=()):
    return {"name": name, "batch": batch, "in_c": in_c, "in_h": h, "in_w": w, "classes": classes, "precision": "fp32",
            "residual_stream": "fp32", "correction": "residual", "stem": stem, "body": body, "segments": [len(body)],
            "coarse": [], "cj_post": "bn_relu",
            "head": {"kind": "gap_mlp" if hidden else "gap_fc", "hidden": list(hidden)}}


C = W.conv_bn_relu
NETS = {
    "widths": _net("widths", 3, 3, 16, 16, [C(20)], [C(33), C(70, k=1, stride=2), C(17, pool=2)], hidden=(72,)),
    "odd_image": _net("odd_image", 2, 1, 9, 11, [W.conv(16, stride=2)], [C(10, pool=2), C(6, k=1)], classes=300),
    "seven_in": _net("seven_in", 5, 7, 12, 8, [C(40, k=1)], [C(64, stride=2), C(65)], hidden=(300,)),
    "seven_in_3x3": _net("seven_in_3x3", 2, 7, 8, 8, [C(12)], [C(16), C(32, pool=2)]),
    "three_in_64": _net("three_in_64", 9, 3, 20, 20, [C(64)], [C(16, k=1)]),
    # the head's K over the CTAs of a cluster (1030: a short last share), ragged tiles
    "wide_head": _net("wide_head", 33, 3, 8, 8, [C(16)], [C(32, k=1)], hidden=(1030, 517)),
    "wide_head_130": _net("wide_head_130", 130, 3, 4, 4, [C(16)], [C(260, k=1)], hidden=(640,), classes=17),
    "one_image": W.tiny_resnet(batch=1),
    "torn": W.tiny_resnet(batch=5),
    "torn_delta": W.tiny_resnet(batch=3, correction="delta"),
}


@pytest.mark.parametrize("name", list(NETS))
def test_small_fp32_networks(name):
    desc = NETS[name]
    _, theta, x, labels = inputs(desc, seed=11)
    report, fails = compare(desc, run_gpu(desc, theta, x, labels), run_oracle(desc, theta, x, labels))
    print(name, {k: f"{v:.1e}" for k, v in report.items()})
    assert not fails, fails
