"""The work a user of this framework has it do, as cases that can be timed and compared.

Kinds of case (key "kind"):
  train   one training step (Algorithm 1, Algorithm 2, SGD) of a parareal network through
          ParaNet.train_step, or through train_step_host from pinned host buffers
  infer   one eval-mode forward pass through ParaNet.infer
  conv    one grouped convolution of a network's layers (forward, data or weight gradient)
          through conv_run
The networks are those of the workload descriptions (VGG-16, ResNet-1001 and its depth-reduced
family, the paper's Parareal ResNet-N, the tiny network); conv cases take the geometry of their
layers or odd sizes around it.

exact() evaluates the same networks and layers in float64 torch from the description and the
parameters drawn here.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import workloads as W
from paper_2103_08802_gb300 import pnn

EPS = 1e-5
# A fixed synthetic batch trained at the paper's 0.1 can diverge within dozens of steps, and a step's
# work does not depend on the rate.
LR = 0.002
# Trained residual branches are small against the stream they are added to; inference nets get
# this gamma on the last BN of every residual branch.
BRANCH_GAMMA = 0.25


# ---------------------------------------------------------------- cases
def listed():
    return [
        # the smallest network: launch latency and the fp32 arithmetic
        {"name": "train_tiny_fp32_b8", "kind": "train", "net": "tiny", "batch": 8, "precision": "fp32", "grads": True},
        # a short bottleneck net at an odd batch, delta correction, fp32 residual stream
        {"name": "train_short_delta_b50", "kind": "train", "net": "resnet", "per_stage": 2, "n": 3, "batch": 50,
         "hw": 32, "classes": 10, "correction": "delta", "stream": "fp32"},
        # Parareal VGG-16 at CIFAR shape: wide 3x3 layers, maxpools, the 4096-wide FC head
        {"name": "train_vgg16_n4_b128", "kind": "train", "net": "vgg16", "batch": 128},
        # Parareal ResNet-1001, 4 subnetworks, CIFAR shape
        {"name": "train_resnet1001_n4_b128", "kind": "train", "net": "resnet", "per_stage": 111, "n": 4, "batch": 128,
         "hw": 32, "classes": 10},
        # 16 subnetworks, 100 classes, fed from host memory as a data loader does
        {"name": "train_resnet1001_n16_host", "kind": "train", "net": "resnet", "per_stage": 111, "n": 16, "batch": 128,
         "hw": 32, "classes": 100, "host": True},
        # the headline workload, and the largest
        {"name": "train_resnet1001_n8_64px", "kind": "train", "net": "resnet", "per_stage": 111, "n": 8, "batch": 256,
         "hw": 64, "classes": 200},
        # evaluation of the headline network at its batch
        {"name": "infer_resnet1001_n8_64px", "kind": "infer", "net": "resnet", "per_stage": 111, "n": 8, "batch": 256,
         "hw": 64, "classes": 200},
        # serving one image
        {"name": "infer_resnet1001_n4_b1", "kind": "infer", "net": "resnet", "per_stage": 111, "n": 4, "batch": 1,
         "hw": 32, "classes": 10},
        # one layer of eight subnetworks in one launch: the bottleneck's expanding 1x1 with residual and
        # BN statistics, the data gradient of its 3x3 with the BN-backward sums, its 3x3's weight gradient
        {"name": "conv_fwd_expand", "kind": "conv", "mode": "forward", "inst": 8, "spread": True, "batch": 256, "hw": 32,
         "c": 16, "k": 64, "ksize": 1, "stride": 1, "res": True, "bn": True},
        {"name": "conv_dgrad_3x3", "kind": "conv", "mode": "dgrad", "inst": 8, "spread": True, "batch": 256, "hw": 32,
         "c": 16, "k": 16, "ksize": 3, "stride": 1, "res": False, "bn": True},
        {"name": "conv_wgrad_3x3", "kind": "conv", "mode": "wgrad", "inst": 8, "spread": True, "batch": 256, "hw": 32,
         "c": 16, "k": 16, "ksize": 3, "stride": 1, "res": False, "bn": True},
        # an odd layer: ragged image, strided, channel counts that fill no tile
        {"name": "conv_fwd_odd_s2", "kind": "conv", "mode": "forward", "inst": 3, "spread": False, "batch": 37, "hw": 27,
         "c": 24, "k": 40, "ksize": 3, "stride": 2, "res": False, "bn": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "infer", "conv", "conv"])
    if kind == "conv":
        spread = rng.random() < 0.5
        c = {"kind": "conv", "mode": rng.choice(["forward", "dgrad", "wgrad"]), "inst": rng.randint(1, 12),
             "spread": spread, "batch": _log(rng, 4, 256), "hw": rng.choice([32, 16]) if spread else rng.randint(4, 40),
             "ksize": rng.choice([1, 3]), "stride": 1 if spread else rng.choice([1, 1, 1, 2])}
        wide = rng.choice([16, 32, 64] if spread else [8, 16, 24, 32, 64, 72, 128])
        c["c"], c["k"] = rng.choice([(wide, wide), (wide, min(4 * wide, 256)), (min(4 * wide, 256), wide)])
        if spread and max(c["c"], c["k"]) > 64:
            c["spread"], c["hw"] = False, 16
        c["res"] = c["mode"] == "forward" and rng.random() < 0.5
        c["bn"] = rng.random() < 0.7
        return c
    if kind == "infer" or rng.random() < 0.7:
        c = {"kind": kind, "net": "resnet", "per_stage": _log(rng, 2, 111), "n": rng.choice([1, 2, 3, 4, 8, 12, 16]),
             "batch": _log(rng, 1 if kind == "infer" else 8, 256), "hw": rng.choice([32, 64]),
             "classes": rng.choice([10, 100, 200])}
        if kind == "train" and rng.random() < 0.3:
            c["net"], c["n"], c["hw"] = "paper", rng.choice([3, 6, 12]), 32
        while c["n"] > c["per_stage"] or 3 * c["per_stage"] <= (c["n"] - 1) * -(-3 * c["per_stage"] // c["n"]):
            c["n"] -= 3 if c["net"] == "paper" else 1
            if c["n"] <= 1:
                c["net"], c["n"] = "resnet", 1
                break
        if kind == "train":
            c["correction"] = rng.choice(["residual", "residual", "delta"])
            c["stream"] = rng.choice(["bf16", "bf16", "fp32"])
            c["host"] = rng.random() < 0.3
        while work(c)["flops"] > 1.9e12:  # no larger than the headline workload
            c["batch"] = c["batch"] * 3 // 4
        return c
    return {"kind": "train", "net": "vgg16", "batch": _log(rng, 8, 256), "correction": rng.choice(["residual", "delta"]),
            "coarse": rng.choice(["one_conv", "paper"]), "host": rng.random() < 0.3}


def _desc(case):
    kw = {"batch": case["batch"], "correction": case.get("correction", "residual")}
    if case["net"] == "tiny":
        d = W.tiny_resnet(precision=case.get("precision", "fp32"), **kw)
    elif case["net"] == "vgg16":
        d = W.parareal_vgg16(coarse=case.get("coarse", "one_conv"), **kw)
    elif case["net"] == "paper":
        d = W.paper_parareal_resnet(case["n"], classes=case["classes"], hw=case["hw"], per_stage=case["per_stage"], **kw)
    else:
        d = W.parareal_resnet1001(n_seg=case["n"], classes=case["classes"], hw=case["hw"], per_stage=case["per_stage"],
                                  **kw)
    if case.get("stream"):
        d["residual_stream"] = case["stream"]
    return d


# ---------------------------------------------------------------- the networks in torch
class _Net:
    """The parareal network of a description.  A walk over it takes parameters in the order of the
    flat vector; `params` is that vector (float64 on the GPU), or None for a dry walk on the meta
    device that records the parameter shapes, the BN layers and the convolutions.  Values are
    (tensor, second moment expected of He-normal weights)."""

    def __init__(self, desc, params=None, running=None):
        self.desc, self.params, self.running = desc, params, running
        self.spec, self.convs, self.bns, self.at, self.rat = [], [], [], 0, 0

    def take(self, kind, *shape):
        if self.params is None:
            self.spec.append((kind, shape))
            return torch.empty(shape, device="meta")
        n = math.prod(shape)
        self.at += n
        return self.params[self.at - n:self.at].view(shape)

    def take_bn(self, c, branch_end=False):
        """(gamma, beta, running mean and variance, position) of one BN layer"""
        g, b = self.take("end_gamma" if branch_end else "gamma", c), self.take("beta", c)
        run = None
        if self.running is not None:
            run = (self.running[self.rat:self.rat + c], self.running[self.rat + c:self.rat + 2 * c])
            self.rat += 2 * c
        self.bns.append([c, 1.0])
        return g, b, run, len(self.bns) - 1, BRANCH_GAMMA ** 2 if branch_end else 1.0

    def bn(self, v, p, relu=True):
        t, m2 = v
        g, b, run, i, out = p
        self.bns[i][1] = m2
        t = F.batch_norm(t, *(run or (None, None)), g, b, training=run is None, momentum=0.0, eps=EPS) \
            if self.params is not None else t
        return (F.relu(t), out / 2) if relu else (t, out)

    def conv(self, v, w, stride=1):
        t, m2 = v
        y = F.conv2d(t, w, stride=stride, padding=w.shape[2] // 2)
        if self.params is None:
            self.convs.append((t.shape[1], t.shape[2] * t.shape[3], y.shape[1], y.shape[2] * y.shape[3], w.shape[2]))
        return y, 2 * m2

    def layer_params(self, s, cin):
        op, c = s["op"], s["cout"]
        if op == "conv":
            return [self.take("w", c, cin, s["k"], s["k"])]
        if op == "conv_bn_relu":
            return [self.take("w", c, cin, s["k"], s["k"]), self.take_bn(c)]
        if op == "basic":
            return [self.take("w", c, cin, 3, 3), self.take_bn(c), self.take("w", c, c, 3, 3), self.take_bn(c)]
        proj = cin != c or s.get("stride", 1) != 1
        if op == "bottleneck":
            m = s["mid"]
            p = [self.take_bn(cin), self.take("w", m, cin, 1, 1), self.take_bn(m), self.take("w", m, m, 3, 3),
                 self.take_bn(m, True), self.take("w", c, m, 1, 1)]
        else:
            p = [self.take_bn(cin), self.take("w", c, cin, 3, 3), self.take_bn(c, True), self.take("w", c, c, 3, 3)]
        return p + ([self.take("w", c, cin, 1, 1)] if proj else [])

    def layer(self, s, v, p):
        op, st = s["op"], s.get("stride", 1)
        if op == "conv":
            return self.conv(v, p[0], st)
        if op == "conv_bn_relu":
            a = self.bn(self.conv(v, p[0], st), p[1])
            return (F.max_pool2d(a[0], 2, 2), 2 * a[1]) if s.get("pool") else a
        if op == "basic":
            z = self.bn(self.conv(self.bn(self.conv(v, p[0]), p[1]), p[2]), p[3], relu=False)
            return F.relu(z[0] + v[0]), (z[1] + v[1]) / 2
        a1 = self.bn(v, p[0])
        if op == "bottleneck":
            h = self.conv(self.bn(self.conv(self.bn(self.conv(a1, p[1]), p[2]), p[3], st), p[4]), p[5])
            wp = p[6:]
        else:
            h = self.conv(self.bn(self.conv(a1, p[1], st), p[2]), p[3])
            wp = p[4:]
        sc = self.conv(a1, wp[0], st) if wp else v
        return h[0] + sc[0], h[1] + sc[1]

    def stack(self, specs, v, ps=None):
        ps = [] if ps is None else list(ps)
        fresh = not ps
        for i, s in enumerate(specs):
            if fresh:
                ps.append(self.layer_params(s, v[0].shape[1]))
            v = self.layer(s, v, ps[i])
        return v, ps

    def forward(self, x):
        d, n = self.desc, len(self.desc["segments"])
        xs, ys, b0 = [], [], 0
        for j in range(n):
            v = (x, 1.0)
            if j == 0:
                v, _ = self.stack(d["stem"], v)
            else:
                c, h = ys[j - 1][0].shape[1:3]
                while v[0].shape[2] > h:
                    v = F.max_pool2d(v[0], 3, 2, 1), 2 * v[1]
                v = self.conv(v, self.take("w", c, v[0].shape[1], 1, 1))
                if d["cj_post"] == "bn_relu":
                    v = self.bn(v, self.take_bn(c))
            xs.append(v)
            y, _ = self.stack(d["body"][b0:b0 + d["segments"][j]], v)
            b0 += d["segments"][j]
            ys.append(y)
        add = lambda a, b, s=1.0: (a[0] + s * b[0], a[1] + b[1])  # noqa: E731
        yt = ys[0]
        if n > 1:
            rs = [add(ys[j], xs[j + 1], -1.0) for j in range(n - 1)]
            rt = rs[0]
            for j in range(n - 1):
                if d["correction"] == "delta":
                    out, ps = self.stack(d["coarse"][j], add(xs[j + 1], rt))
                    out = add(out, self.stack(d["coarse"][j], xs[j + 1], ps)[0], -1.0)
                else:
                    out, _ = self.stack(d["coarse"][j], rt)
                rt = add(rs[j + 1], out) if j + 1 < n - 1 else out
            yt = add(ys[n - 1], rt)
        if d["head"]["kind"] == "bn_relu_gap_fc":
            yt = self.bn(yt, self.take_bn(yt[0].shape[1]))
        f = yt[0].mean(dim=(2, 3))
        widths = [f.shape[1]] + list(d["head"]["hidden"]) + [d["classes"]]
        for i in range(len(widths) - 1):
            f = F.linear(f, self.take("w", widths[i + 1], widths[i]), self.take("beta", widths[i + 1]))
            if i < len(widths) - 2:
                f = F.relu(f)
        return f


def _dry(desc):
    net = _Net(desc)
    with torch.no_grad():
        net.forward(torch.empty((1, desc["in_c"], desc["in_h"], desc["in_w"]), device="meta"))
    return net


def _theta(desc, seed, infer):
    """He-normal weights, BN gamma 1 (inference: small ends of the residual branches), beta and bias 0."""
    net = _dry(desc)
    g = torch.Generator("cuda").manual_seed(seed)
    parts = []
    for kind, shape in net.spec:
        n = math.prod(shape)
        if kind == "w":
            parts.append(torch.randn(n, generator=g, device="cuda") * math.sqrt(2.0 / math.prod(shape[1:])))
        elif kind == "beta":
            parts.append(torch.zeros(n, device="cuda"))
        else:
            parts.append(torch.full((n,), BRANCH_GAMMA if infer and kind == "end_gamma" else 1.0, device="cuda"))
    return net, torch.cat(parts)


def _running(net):
    """Running means 0 and the variances that He-normal weights give each BN's input."""
    return torch.cat([torch.cat([torch.zeros(c), torch.full((c,), v)]) for c, v in net.bns])


def _batch(desc, seed):
    g = torch.Generator("cuda").manual_seed(seed + 7919)
    x = torch.randn((desc["batch"], desc["in_c"], desc["in_h"], desc["in_w"]), generator=g, device="cuda")
    if desc["precision"] == "bf16":
        x = x.bfloat16().float()
    labels = torch.randint(0, desc["classes"], (desc["batch"],), generator=g, device="cuda", dtype=torch.int32)
    return x, labels


# ---------------------------------------------------------------- one grouped convolution
def _geometry(case):
    out = []
    for i in range(case["inst"]):
        s = i * 3 // case["inst"] if case["spread"] else 0  # the stage: half the size, twice the channels
        out.append({"batch": case["batch"], "h": case["hw"] >> s, "w": case["hw"] >> s, "c": case["c"] << s,
                    "k": case["k"] << s, "ksize": case["ksize"], "stride": case["stride"]})
    return out


def _conv_inputs(case, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    insts = []
    for d in _geometry(case):
        b, h, w, c, k, r, st = (d[n] for n in ("batch", "h", "w", "c", "k", "ksize", "stride"))
        p, q = (h - 1) // st + 1, (w - 1) // st + 1
        i = dict(d)
        i["wt"] = (rnd(k, r, r, c) * math.sqrt(2.0 / (r * r * c))).bfloat16()
        if case["mode"] != "dgrad" or case["bn"]:
            i["x"] = (rnd(b, h, w, c) + 0.3 * rnd(c)).bfloat16()
        if case["bn"]:  # the BN(+ReLU) in front of the layer
            i["bn_scale"], i["bn_shift"], i["relu"] = 0.5 + torch.rand(c, generator=g, device="cuda"), 0.3 * rnd(c), 1
        if case["mode"] == "forward":
            i["y"] = torch.empty(b, p, q, k, dtype=torch.bfloat16, device="cuda")
            if case["res"]:
                i["res"] = rnd(b, p, q, k).bfloat16()
            i["y_mean"], i["y_rstd"] = torch.empty(k, device="cuda"), torch.empty(k, device="cuda")
        else:
            i["dy"] = rnd(b, p, q, k) * 1e-3
            if case["mode"] == "dgrad":
                i["dx"] = torch.empty(b, h, w, c, device="cuda")
                if case["bn"]:
                    xf = i["x"].float().view(-1, c)
                    i["bn_mean"], i["bn_rstd"] = xf.mean(0), (xf.var(0, unbiased=False) + EPS).rsqrt()
                    i["dgamma"], i["dbeta"] = torch.empty(c, device="cuda"), torch.empty(c, device="cuda")
            else:
                i["dw"] = torch.empty(k, r, r, c, device="cuda")
        insts.append(i)
    return insts


CONV_OUT = {"forward": ("y", "y_mean", "y_rstd"), "dgrad": ("dx", "dgamma", "dbeta"), "wgrad": ("dw",)}


def _conv_exact(case, i):
    nchw = lambda t: t.double().permute(0, 3, 1, 2)  # noqa: E731
    wt = nchw(i["wt"])
    pad, st, out = case["ksize"] // 2, case["stride"], {}
    v = None
    if "x" in i:
        v = nchw(i["x"])
        if case["bn"]:
            pre = v * i["bn_scale"].double().view(1, -1, 1, 1) + i["bn_shift"].double().view(1, -1, 1, 1)
            v = F.relu(pre)
    if case["mode"] == "forward":
        y = F.conv2d(v, wt, stride=st, padding=pad)
        if case["res"]:
            y = y + nchw(i["res"])
        out["y"] = y.permute(0, 2, 3, 1).contiguous()
        out["y_mean"] = y.mean(dim=(0, 2, 3))
        out["y_rstd"] = (y.var(dim=(0, 2, 3), unbiased=False) + EPS).rsqrt()
        return out
    dy = nchw(i["dy"])
    if case["mode"] == "wgrad":
        wt = wt.clone().requires_grad_()
        F.conv2d(v, wt, stride=st, padding=pad).backward(dy)
        out["dw"] = wt.grad.permute(0, 2, 3, 1).contiguous()
        return out
    z = torch.zeros((i["batch"], i["c"], i["h"], i["w"]), dtype=torch.float64, device="cuda", requires_grad=True)
    F.conv2d(z, wt, stride=st, padding=pad).backward(dy)
    out["dx"] = z.grad.permute(0, 2, 3, 1).contiguous()
    if case["bn"]:
        g = z.grad * (pre > 0)
        xhat = (nchw(i["x"]) - i["bn_mean"].double().view(1, -1, 1, 1)) * i["bn_rstd"].double().view(1, -1, 1, 1)
        out["dgamma"], out["dbeta"] = (g * xhat).sum(dim=(0, 2, 3)), g.sum(dim=(0, 2, 3))
    return out


# ---------------------------------------------------------------- the interface
def prepare(case, seed):
    if case["kind"] == "conv":
        return {"case": case, "insts": _conv_inputs(case, seed)}
    desc = _desc(case)
    infer = case["kind"] == "infer"
    dry, theta = _theta(desc, seed, infer)
    net = pnn.ParaNet(desc, lr=LR, inference=infer)
    net.set_params(theta.cpu().numpy())
    x, labels = _batch(desc, seed)
    s = {"case": case, "net": net, "x": x}
    if infer:
        net.set_running_stats(_running(dry).numpy())
        s["logits"] = torch.empty((desc["batch"], desc["classes"]), device="cuda")
        return s
    # the workspace is the caller's; it begins with the parameters, then their gradients (each
    # region 256-byte aligned; convolution weights as [K][R][S][C])
    n = theta.numel()
    at = (4 * n + 255) // 256 * 256
    s["params"] = net.ws[:4 * n].view(torch.float32)
    s["grads"] = net.ws[at:at + 4 * n].view(torch.float32)
    if case.get("host"):
        s["x"], s["labels"] = x.cpu().pin_memory(), labels.cpu().pin_memory()
    else:
        s["labels"], s["loss"] = labels, torch.zeros(1, device="cuda")
    return s


def run(state):
    case = state["case"]
    if case["kind"] == "conv":
        insts = state["insts"]
        pnn.conv_run(case["mode"], insts)
        return [{n: i[n] for n in CONV_OUT[case["mode"]] if n in i} for i in insts]
    if case["kind"] == "infer":
        state["net"].infer(state["x"], state["logits"])
        return {"logits": state["logits"]}
    if case.get("host"):
        loss = state["net"].train_step_host(state["x"], state["labels"])
    else:
        state["net"].train_step(state["x"], state["labels"], state["loss"])
        loss = state["loss"]
    out = {"loss": loss, "params": state["params"]}
    if case.get("grads"):
        out["grads"] = state["grads"]
    return out


def work(case):
    """Every convolution's operands read and results written once (activations in their storage type,
    gradients and parameters in fp32), and its multiply-adds."""
    if case["kind"] == "conv":
        fl = by = 0
        for d in _geometry(case):
            st = d["stride"]
            m_in, m_out = d["batch"] * d["h"] * d["w"], d["batch"] * ((d["h"] - 1) // st + 1) * ((d["w"] - 1) // st + 1)
            nw = d["c"] * d["k"] * d["ksize"] ** 2
            fl += 2 * m_out * nw
            if case["mode"] == "forward":
                by += 2 * m_in * d["c"] + 2 * m_out * d["k"] * (2 if case["res"] else 1) + 2 * nw
            elif case["mode"] == "dgrad":
                by += 4 * m_out * d["k"] + (6 if case["bn"] else 4) * m_in * d["c"] + 2 * nw
            else:
                by += 2 * m_in * d["c"] + 4 * m_out * d["k"] + 4 * nw
        return {"bytes": by, "flops": fl}
    desc = _desc(case)
    net = _dry(desc)
    b, e = desc["batch"], 2 if desc["precision"] == "bf16" else 4
    fl = by = 0
    for ci, mi, co, mo, k in net.convs:
        fl += 2 * b * mo * co * ci * k * k
        by += e * b * (mi * ci + mo * co)
        if case["kind"] == "train":
            fl += 4 * b * mo * co * ci * k * k
            by += b * (e * mi * ci + 4 * mo * co + 4 * mi * ci)
    n = sum(math.prod(s) for _, s in net.spec)
    by += 4 * n * (5 if case["kind"] == "train" else 1) + 4 * b * desc["in_c"] * desc["in_h"] * desc["in_w"]
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """About four times the difference between the TMA-fed and the thread-gathered convolutions (other
    orders of the same fp32 sums).  A deep bf16 network amplifies a flipped rounding: its loss moved by
    1e-3 and its updated parameters by 2e-3 at a learning rate of 0.01, a VGG's parameters by 2e-4."""
    if case["kind"] == "conv":
        # bf16 outputs: a sum next to a rounding boundary moves by one unit in the last place
        return {"rel": 5e-4, "max": 0.02} if case["mode"] == "forward" else {"rel": 1e-5}
    if case["kind"] == "infer":
        return {"rel": 0.01}
    if case["net"] == "tiny":
        return {"rel": 1e-5}
    return {"rel": 1e-3} if case["net"] == "vgg16" or case["per_stage"] <= 3 else {"rel": 0.02}


def exact(case, seed):
    if case["kind"] == "conv":
        out = []
        for i in _conv_inputs(case, seed):
            e = _conv_exact(case, i)
            out.append({n: e[n] for n in CONV_OUT[case["mode"]] if n in i})
        return out
    desc = _desc(case)
    w = work(case)
    if w["flops"] > (2e12 if case["kind"] == "infer" else 3e11):
        return None  # too long in float64
    infer = case["kind"] == "infer"
    dry, theta = _theta(desc, seed, infer)
    x, labels = _batch(desc, seed)
    if infer:
        net = _Net(desc, theta.double(), _running(dry).cuda().double())
        with torch.no_grad():
            return {"logits": torch.cat([_rewind(net).forward(c.double()) for c in x.split(32)])}
    p = theta.double().requires_grad_()
    loss = F.cross_entropy(_Net(desc, p).forward(x.double()), labels.long())
    loss.backward()
    step = p.grad + 5e-4 * p.detach()  # weight decay, then Nesterov momentum 0.9 from zero
    new = p.detach() - LR * (step + 0.9 * step)
    out = {"loss": loss.item() if case.get("host") else loss.detach().view(1), "params": _internal(dry, new)}
    if case.get("grads"):
        out["grads"] = _internal(dry, p.grad)
    return out


def _rewind(net):
    net.at = net.rat = 0
    net.bns.clear()
    return net


def _internal(dry, flat):
    """The flat vector with convolution weights as [K][R][S][C]."""
    parts, at = [], 0
    for _, shape in dry.spec:
        t = flat[at:at + math.prod(shape)]
        at += t.numel()
        parts.append(t.view(shape).permute(0, 2, 3, 1).reshape(-1) if len(shape) == 4 else t)
    return torch.cat(parts)
