"""Streaming convolution of layers with 128, 192 or 256 output channels, 64 per
CTA, against FP64 on the same BF16 operands: resident and travelling weights,
one and two input tensors, ragged rows and columns, segments of 2 rows (variant
5) and of 16 and more (the default choice), a channel slice of a wider output."""

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


@pytest.mark.parametrize("n,h,w,c0,c1,cout,variant", [
    (1, 700, 200, 64, 0, 128, 0), (1, 611, 128, 128, 128, 128, 0), (1, 37, 256, 64, 0, 128, 5),
    (1, 64, 300, 96, 32, 192, 5), (2, 33, 130, 32, 128, 256, 5), (3, 2, 128, 32, 0, 256, 5)])
def test_grouped_streaming_layer(lib, n, h, w, c0, c1, cout, variant):
    import torch
    g = torch.Generator(device="cuda").manual_seed(h * w + cout)
    cin, pad = c0 + c1, 32

    def vp(t):
        return C.c_void_p(t.data_ptr()) if t is not None else None

    x0 = torch.randn((n, h, w, c0), generator=g, device="cuda").to(torch.bfloat16)
    x1 = torch.randn((n, h, w, c1), generator=g, device="cuda").to(torch.bfloat16) if c1 else None
    wf = (torch.randn((cout, cin, 3, 3), generator=g, device="cuda") * math.sqrt(2.0 / (9 * cin))).contiguous()
    b = torch.randn(cout, generator=g, device="cuda") * 0.1
    wt = torch.empty(9 * cout * cin, dtype=torch.bfloat16, device="cuda")
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.glbm_nn_tc_pack_weights(vp(wf), cout, cin, 3, cout, cin, vp(wt), st) == 0
    y = torch.full((n, h, w, cout + pad), -7.0, dtype=torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    lib.glbm_nn_tc_set_variant(variant)
    rc = lib.glbm_nn_tc_conv(vp(x0), c0, vp(x1), c1, n, h, w, 3, vp(wt), vp(b), cout, vp(y), cout + pad, 1, 0, 0,
                             vp(err), st)
    lib.glbm_nn_tc_set_variant(0)
    assert rc == 0
    torch.cuda.synchronize()
    assert int(err) == 0
    x = x0 if x1 is None else torch.cat([x0, x1], 3)
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), wf.to(torch.bfloat16).double(), b.double(),
                                     padding=1).relu().permute(0, 2, 3, 1)
    got = y[..., :cout].double()
    # the BF16 output rounding (half an ulp = 2^-9 relative) plus FP32 accumulation
    assert bool(((got - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-6 * ref.abs().max()).all())
    assert bool((y[..., cout:] == -7.0).all())


@pytest.mark.parametrize("n,h,w,c0,c1,cout,variant", [
    (1, 640, 256, 128, 0, 128, 0), (1, 611, 130, 64, 0, 128, 0), (1, 37, 200, 32, 64, 192, 5),
    (2, 2, 128, 64, 64, 256, 5), (1, 65, 129, 32, 0, 128, 5), (1, 256, 256, 128, 0, 128, 0),
    (1, 128, 256, 64, 0, 128, 0), (2, 101, 130, 32, 0, 192, 0)])
def test_resident_groups_sum_in_the_tile_kernels_order(lib, n, h, w, c0, c1, cout, variant):
    """Up to 128 input channels the groups add taps and channels in the order of
    the tile kernel (variant 1): the outputs are its bits."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(h * w + cout)
    cin = c0 + c1

    def vp(t):
        return C.c_void_p(t.data_ptr()) if t is not None else None

    x0 = torch.randn((n, h, w, c0), generator=g, device="cuda").to(torch.bfloat16)
    x1 = torch.randn((n, h, w, c1), generator=g, device="cuda").to(torch.bfloat16) if c1 else None
    wf = torch.randn((cout, cin, 3, 3), generator=g, device="cuda").contiguous()
    b = torch.randn(cout, generator=g, device="cuda")
    wt = torch.empty(9 * cout * cin, dtype=torch.bfloat16, device="cuda")
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.glbm_nn_tc_pack_weights(vp(wf), cout, cin, 3, cout, cin, vp(wt), st) == 0
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = []
    for v in (1, variant):
        y = torch.full((n, h, w, cout), -7.0, dtype=torch.bfloat16, device="cuda")
        lib.glbm_nn_tc_set_variant(v)
        rc = lib.glbm_nn_tc_conv(vp(x0), c0, vp(x1), c1, n, h, w, 3, vp(wt), vp(b), cout, vp(y), cout, 0, 0, 0, vp(err),
                                 st)
        lib.glbm_nn_tc_set_variant(0)
        assert rc == 0
        torch.cuda.synchronize()
        assert int(err) == 0
        out.append(y)
    assert torch.equal(*out)
