"""Which kernels a grouped convolution takes by itself (pnn_conv_kernel, host only):
every case of test_gpu_auto_conv_kernels is one that the 1x1, 3x3 and
weight-gradient kernels take, and a step past each edge of their rules is not."""
import ctypes as C

import pytest

import test_gpu_auto_conv_kernels as A

GATHERED, TMA, POINTWISE, C3X3, WGRAD = range(5)


@pytest.fixture(scope="module")
def lib():
    from paper_2103_08802_gb300 import build, pnn
    build.build()
    return pnn.load()


def kernel(lib, mode, specs, impl=0, bn_offset=0, offset=0, y_fp32=False, res_fp32=False, bn_sums=True):
    from paper_2103_08802_gb300 import pnn
    arr = (pnn.ConvArgs * len(specs))()
    for a, s in zip(arr, specs):
        for key in ("batch", "h", "w", "c", "k", "ksize", "stride"):
            setattr(a, key, s[key])
        a.x = a.wt = a.y = a.dy = a.dx = a.dw = 4096 + offset  # never dereferenced
        a.x_dtype = 0 if s.get("x_fp32") else 1
        a.y_dtype, a.res_dtype = (0 if y_fp32 else 1), (0 if res_fp32 else 1)
        a.res = 4096 if res_fp32 else None
        if s.get("bn"):
            a.bn_scale = a.bn_shift = 4096 + bn_offset
            if mode == 1 and bn_sums:
                a.bn_mean = a.bn_rstd = 4096 + bn_offset
                a.dgamma = a.dbeta = 4096
    out = C.c_int32()
    assert lib.pnn_conv_kernel(mode, impl, len(specs), arr, C.byref(out)) == 0
    return out.value


def _specs(v):
    return v if isinstance(v, list) else [v]


@pytest.mark.parametrize("name", list(A.PW))
def test_pointwise_cases(lib, name):
    assert kernel(lib, 0, _specs(A.PW[name])) == POINTWISE
    # (a data gradient reads an fp32 BN input in the older kernels only)
    fp32 = any(s.get("x_fp32") for s in _specs(A.PW[name]))
    assert kernel(lib, 1, _specs(A.PW[name])) == (TMA if fp32 else POINTWISE)


@pytest.mark.parametrize("name", list(A.C3))
def test_3x3_cases(lib, name):
    assert kernel(lib, 0, _specs(A.C3[name])) == C3X3
    if not any(s.get("x_fp32") for s in _specs(A.C3[name])):
        assert kernel(lib, 1, _specs(A.C3[name])) == C3X3


@pytest.mark.parametrize("name", list(A.WG))
def test_weight_gradient_cases(lib, name):
    assert kernel(lib, 2, _specs(A.WG[name])) == WGRAD


P = dict(batch=2, h=16, w=16, c=16, k=64, ksize=1, stride=1, bn=True)
T = dict(batch=2, h=16, w=16, c=16, k=32, ksize=3, stride=1, bn=True)


@pytest.mark.parametrize("mode,spec,kw", [
    (0, dict(P, stride=2), {}), (0, dict(P, c=24), {}), (0, dict(P, c=320), {}), (0, dict(P, k=48), {}),
    (0, dict(P, c=128, k=128), {}), (0, P, dict(y_fp32=True)), (0, P, dict(res_fp32=True)), (0, P, dict(impl=1)),
    (0, P, dict(impl=2)), (0, P, dict(bn_offset=4)), (0, P, dict(offset=8)), (1, dict(P, x_fp32=True), {}),
    (1, P, dict(bn_offset=4)), (0, dict(T, stride=2), {}), (0, dict(T, c=24), {}), (0, dict(T, c=96), {}),
    (0, dict(T, h=14, w=14), {}), (0, dict(T, h=8, w=16), {}), (0, dict(T, h=8, w=8, batch=3, c=48), {}),
    (0, T, dict(y_fp32=True)), (1, dict(T, x_fp32=True), {}), (2, dict(P, stride=2), {}), (2, dict(P, c=128, k=128), {}),
    (2, dict(P, c=48), {}), (2, dict(T, w=64, h=16), {}), (2, dict(T, c=24), {}), (2, dict(T, k=96), {}),
    (2, dict(T, h=14, w=14), {}), (2, T, dict(bn_offset=4)),
])
def test_past_the_edges(lib, mode, spec, kw):
    assert kernel(lib, mode, [spec], **kw) in (GATHERED, TMA)


def test_one_instance_outside_takes_the_group_out(lib):
    assert kernel(lib, 0, [P, P]) == POINTWISE and kernel(lib, 0, [P, dict(P, k=48)]) in (GATHERED, TMA)
    assert kernel(lib, 0, [P, T]) in (GATHERED, TMA) and kernel(lib, 2, [P, T]) in (GATHERED, TMA)
