"""Layers with 128, 192 or 256 output channels give the same bits whichever
kernel the sizes pick: the streaming kernel's groups add taps and channels in
the order of the tile kernel (variant 1), and inputs too wide for that order
stay on the tile kernel.  Input widths on both sides of the line, by default
and with streaming asked for, ragged rows and columns."""

import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_1601_00704_gb300 import build
    build.build()
    import paper_1601_00704_gb300 as p
    return p.load()


def _vp(t):
    return C.c_void_p(t.data_ptr()) if t is not None else None


@pytest.mark.parametrize("n,h,w,c0,c1,cout,variant", [
    (1, 512, 512, 128, 128, 128, 0), (1, 611, 130, 128, 64, 128, 0), (1, 700, 128, 96, 64, 256, 0),
    (1, 37, 300, 224, 0, 192, 5), (2, 33, 130, 128, 128, 256, 5), (1, 2, 128, 160, 0, 128, 5), (1, 65, 129, 96, 96, 128, 5),
    (1, 40, 256, 128, 128, 192, 5), (1, 600, 128, 160, 128, 128, 0), (1, 300, 256, 64, 64, 128, 0),
    (4, 24, 650, 64, 64, 256, 0), (3, 24, 650, 32, 0, 192, 0)])
def test_grouped_layers_have_the_tile_kernels_bits(lib, n, h, w, c0, c1, cout, variant):
    import torch
    g = torch.Generator(device="cuda").manual_seed(h * w + c0 + cout)
    cin = c0 + c1
    x0 = torch.randn((n, h, w, c0), generator=g, device="cuda").to(torch.bfloat16)
    x1 = torch.randn((n, h, w, c1), generator=g, device="cuda").to(torch.bfloat16) if c1 else None
    wf = torch.randn((cout, cin, 3, 3), generator=g, device="cuda").contiguous()
    b = torch.randn(cout, generator=g, device="cuda")
    wt = torch.empty(9 * cout * cin, dtype=torch.bfloat16, device="cuda")
    st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.glbm_nn_tc_pack_weights(_vp(wf), cout, cin, 3, cout, cin, _vp(wt), st) == 0
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = []
    for v in (1, variant):
        y = torch.full((n, h, w, cout), -7.0, dtype=torch.bfloat16, device="cuda")
        lib.glbm_nn_tc_set_variant(v)
        rc = lib.glbm_nn_tc_conv(_vp(x0), c0, _vp(x1), c1, n, h, w, 3, _vp(wt), _vp(b), cout, _vp(y), cout, 0, 0, 0,
                                 _vp(err), st)
        lib.glbm_nn_tc_set_variant(0)
        assert rc == 0
        torch.cuda.synchronize()
        assert int(err) == 0
        out.append(y)
    assert torch.equal(*out)
