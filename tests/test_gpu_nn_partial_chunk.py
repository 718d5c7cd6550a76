"""Streaming convolution of inputs whose last 32-channel chunk is half empty
(48, 80 and 112 channels) against FP64 on the same BF16 operands, by default
choice (segments of 16 rows and more) and with streaming asked for."""

import ctypes as C
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    return p.load()


def _vp(t):
    return C.c_void_p(t.data_ptr())


@pytest.mark.parametrize("up2", [False, True])
@pytest.mark.parametrize("n,h,w,variant", [(1, 2600, 128, 0), (2, 37, 200, 5)])
@pytest.mark.parametrize("c0,cout", [(16, 32), (48, 32), (48, 64), (80, 32), (80, 64), (112, 32), (112, 64)])
def test_half_empty_last_chunk(lib, n, h, w, variant, c0, cout, up2):
    import torch
    g = torch.Generator(device="cuda").manual_seed(c0 + cout)
    x = torch.randn((n, h, w, c0), generator=g, device="cuda").to(torch.bfloat16)
    wf = (torch.randn((cout, c0, 3, 3), generator=g, device="cuda") * math.sqrt(2.0 / (9 * c0))).contiguous()
    b = torch.randn(cout, generator=g, device="cuda") * 0.1
    wt = torch.empty(9 * cout * c0, dtype=torch.bfloat16, device="cuda")
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.glbm_nn_tc_pack_weights(_vp(wf), cout, c0, 3, cout, c0, _vp(wt), st) == 0
    f = 2 if up2 else 1
    y = torch.full((n, f * h, f * w, cout), -7.0, dtype=torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    lib.glbm_nn_tc_set_variant(variant)
    if up2:
        rc = lib.glbm_nn_tc_conv_up2(_vp(x), c0, None, 0, n, h, w, _vp(wt), _vp(b), cout, _vp(y), cout, 1, _vp(err), st)
    else:
        rc = lib.glbm_nn_tc_conv(_vp(x), c0, None, 0, n, h, w, 3, _vp(wt), _vp(b), cout, _vp(y), cout, 1, 0, 0, _vp(err),
                                 st)
    lib.glbm_nn_tc_set_variant(0)
    if up2 and rc != 0:
        assert rc == -1  # weights beyond shared memory: refused, and nothing is written
        assert bool((y == -7.0).all())
        return
    assert rc == 0
    torch.cuda.synchronize()
    assert int(err) == 0
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), wf.to(torch.bfloat16).double(), b.double(),
                                     padding=1).relu()
    if up2:
        ref = ref.repeat_interleave(2, 2).repeat_interleave(2, 3)
    ref = ref.permute(0, 2, 3, 1)
    # the BF16 output rounding (half an ulp = 2^-9 relative) plus FP32 accumulation
    assert bool(((y.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-6 * ref.abs().max()).all())
