"""The tensor-core convolution kernels at the edges of their tilings, against
the FP64 reference: image heights and widths that leave partial 128-pixel tiles
of the padded image, strips of wide images, channel counts that pick each
weight-block and K-group variant, and pixel splits of the weight gradient that
end inside a column, leave one row, or go through a cluster.

Bounds: outputs are rounded to BF16 once (2^-9 of each value, so below 4e-3 in
relative L2); the FP32 sums of the weight gradient run over at most 2^18 terms
in blocks of 16, an error of a few 1e-6 of the result: 2e-5."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

SIZES = [  # n, ci, co, h, w
    (1, 16, 32, 4, 32), (3, 32, 32, 4, 160), (2, 48, 64, 12, 96), (1, 64, 96, 8, 128), (2, 32, 192, 4, 256),
    (1, 96, 32, 20, 512), (2, 64, 128, 4, 320), (1, 128, 64, 8, 640), (5, 256, 128, 4, 64), (1, 32, 96, 64, 128),
    (4, 128, 256, 4, 32), (9, 32, 64, 32, 128), (1, 160, 32, 4, 384),
]


@pytest.mark.parametrize("n,ci,co,h,w", SIZES)
def test_convolution_and_gradients(n, ci, co, h, w):
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import surrogate
    lib = surrogate.load_unet()
    g = t.Generator("cuda").manual_seed(n + ci + co + h + w)
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    vp = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    x = t.randn((n, h, w, ci), generator=g, device="cuda").bfloat16()
    dy = t.randn((n, h, w, co), generator=g, device="cuda").bfloat16()
    wt = (t.randn((co, ci, 3, 3), generator=g, device="cuda") * (2 / (9 * ci)) ** 0.5).bfloat16().float()
    b = t.randn(co, generator=g, device="cuda")
    xr = x.double().permute(0, 3, 1, 2).contiguous().requires_grad_(True)
    wr = wt.double().requires_grad_(True)
    xp = t.nn.functional.pad(t.cat([xr[..., -1:], xr, xr[..., :1]], -1), (0, 0, 1, 1))
    ref = sum(t.einsum("oi,nihw->nohw", wr[:, :, i, j], xp[:, :, i:i + h, j:j + w]) for i in range(3) for j in range(3))
    ref.backward(dy.double().permute(0, 3, 1, 2))
    rel = lambda a, r: float(t.linalg.norm(a.double() - r) / t.linalg.norm(r))  # noqa: E731

    pk = t.empty(int(lib.unet_conv_pack_elems(co, ci, 0)), dtype=t.bfloat16, device="cuda")
    assert lib.unet_conv_pack(vp(wt), co, ci, 0, vp(pk), s) == 0
    y = t.empty_like(dy)
    assert lib.unet_conv3x3(vp(x), ci, ci, vp(pk), vp(b), vp(y), co, co, n, h, w, 1, s) == 0
    assert rel(y.permute(0, 3, 1, 2), t.relu(ref.detach() + b.double()[None, :, None, None])) < 4e-3
    if ci % 32 == 0:
        pk = t.empty(int(lib.unet_conv_pack_elems(co, ci, 1)), dtype=t.bfloat16, device="cuda")
        assert lib.unet_conv_pack(vp(wt), co, ci, 1, vp(pk), s) == 0
        dx = t.empty_like(x)
        assert lib.unet_conv3x3(vp(dy), co, co, vp(pk), None, vp(dx), ci, ci, n, h, w, 0, s) == 0
        assert rel(dx.permute(0, 3, 1, 2), xr.grad) < 4e-3
    dw = t.zeros((co, ci, 3, 3), device="cuda")
    assert lib.unet_conv3x3_bwd_weight(vp(x), ci, ci, vp(dy), co, co, vp(dw), None, n, h, w, s) == 0
    assert rel(dw, wr.grad) < 2e-5
    assert lib.unet_tc_error(s, 1) == 0


@pytest.mark.parametrize("h", [1, 2, 3])
def test_weight_gradient_of_one_to_three_rows(h):
    """Tap rows that never meet the image contribute nothing."""
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import surrogate
    lib = surrogate.load_unet()
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    g = t.Generator("cuda").manual_seed(h)
    n, c, w = 2, 32, 16
    x = t.randn((n, h, w, c), generator=g, device="cuda").bfloat16()
    dy = t.randn((n, h, w, c), generator=g, device="cuda").bfloat16()
    dw = t.zeros((c, c, 3, 3), device="cuda")
    vp = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    assert lib.unet_conv3x3_bwd_weight(vp(x), c, c, vp(dy), c, c, vp(dw), None, n, h, w, s) == 0
    xd, d = x.double().permute(0, 3, 1, 2), dy.double().permute(0, 3, 1, 2)
    xp = t.nn.functional.pad(t.cat([xd[..., -1:], xd, xd[..., :1]], -1), (0, 0, 1, 1))
    ref = t.stack([t.stack([t.einsum("nohw,nihw->oi", d, xp[:, :, i:i + h, j:j + w]) for j in range(3)], -1)
                   for i in range(3)], -2)
    assert float(t.linalg.norm(dw.double() - ref) / t.linalg.norm(ref)) < 2e-5
    assert t.all(dw[ref == 0] == 0)
