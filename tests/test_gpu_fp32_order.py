"""An fp32 (check mode) network adds in a fixed order, so its results keep their
bits whatever tiles, splits and loads in flight its kernels use: gradients of one
step, parameters and BN running statistics after three, logits of an inference
pass, as digests of their fp32 bytes.  The recorded digests are those of the first
CUDA-core kernels.  (A sum in another order moves a BN statistic by a last bit; one
pre-activation next to zero that changes sides of its ReLU then moves the gradients
by 1e-5 to 1e-3.)

The networks: the tiny one at its batch and others, and those of
test_gpu_simt_kernels, for the widths on both sides of the tiles, ragged rows, heads
with a long K; layers wider than 256 channels; more partial tiles than one round of
the BN finalisation takes."""
import hashlib
import json
import os

import numpy as np
import pytest

import workloads as W
from test_gpu_simt_kernels import C, NETS, _net

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "fp32_step_digests.json")

CASES = {f"tiny_seed{s}": (W.tiny_resnet(batch=8), s) for s in range(4)}
CASES.update({n: (d, 11) for n, d in NETS.items()})
CASES["wide512"] = (_net("wide512", 5, 3, 8, 8, [C(16)], [W.basic(16), C(512), W.basic(512)]), 11)
CASES["ragged_rows"] = (_net("ragged_rows", 19, 3, 20, 20, [C(24)], [C(16, k=1), C(48), C(200)]), 11)
CASES["many_tiles"] = (_net("many_tiles", 140, 3, 32, 32, [C(16)], [C(16, k=1), C(40, k=1)]), 11)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2103_08802_gb300 import build
    build.build()


def digests(desc, seed):
    import torch
    from paper_2103_08802_gb300 import pnn
    sha = lambda *a: hashlib.sha256(b"".join(np.ascontiguousarray(v).tobytes() for v in a)).hexdigest()[:16]  # noqa: E731
    rng = np.random.Generator(np.random.PCG64(seed))
    net = pnn.ParaNet(desc, lr=0.002)
    spec, n = net.param_spec(), net.num_params
    theta = np.zeros(n, np.float32)
    for (kind, dims, at), end in zip(spec, [s[2] for s in spec[1:]] + [n]):
        fan = max(1, int(np.prod([v for v in dims[1:] if v > 0])))
        noise = rng.standard_normal(end - at)
        theta[at:end] = 1 + 0.1 * noise if kind == 1 else 0.1 * noise if kind == 2 else noise * np.sqrt(2.0 / fan)
    x = rng.standard_normal((desc["batch"], desc["in_c"], desc["in_h"], desc["in_w"])).astype(np.float32)
    labels = rng.integers(0, desc["classes"], desc["batch"]).astype(np.int32)
    out = {"inputs": sha(theta, x, labels)}
    xd, ld, loss = torch.from_numpy(x).cuda(), torch.from_numpy(labels).cuda(), torch.zeros(1, device="cuda")
    net.set_params(theta)
    net.forward(xd, ld, loss)
    net.backward()
    net.sync()
    out["grads"] = sha(loss.cpu().numpy(), net.get_tensor("logits"), net.get_grads())
    net.set_params(theta)
    for _ in range(3):
        net.train_step(xd, ld, loss)
    net.sync()
    run = net.running_stats()
    out["steps"] = sha(loss.cpu().numpy(), net.get_params(), run)
    net.close()
    net = pnn.ParaNet(desc, inference=True)
    net.set_params(theta)
    net.set_running_stats(run)
    logits = torch.empty((desc["batch"], desc["classes"]), device="cuda")
    net.infer(xd, logits)
    net.sync()
    out["infer"] = sha(logits.cpu().numpy())
    net.close()
    return out


@pytest.mark.parametrize("name", list(CASES))
def test_results_keep_their_bits(name):
    want = json.load(open(GOLDEN))[name]
    got = digests(*CASES[name])
    assert got["inputs"] == want["inputs"], "the seeded inputs are not those of the recorded digests"
    assert got == want
