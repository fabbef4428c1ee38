"""Accuracy of the weight gradient on large batches, against 64 bits, where all
products are positive and the error of the FP32 sums adds up.

An accumulator takes at most 4096 pixels, 16 a matrix instruction: 256 additions,
each off by less than one unit in the last place (2^-23) of a running sum that
is half the total on average, so 2^-16 in all (1.6e-5). The partial sums are
rounded to nearest: N addends, 2^-24 of half the total each, N / 2^25; with
N = n h w / 4096 rounded up to whole waves of 152 CTAs (304 for at most 16
channels), below 1000 here, 3e-5."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ci,co,h,w", [(160, 32, 32, 64, 256), (160, 192, 64, 32, 128), (400, 16, 32, 32, 256),
                                         (96, 64, 32, 96, 96), (90, 24, 32, 100, 240)])
def test_long_sums(n, ci, co, h, w):
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import surrogate
    lib = surrogate.load_unet()
    vp = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    g = t.Generator("cuda").manual_seed(n)
    x = (t.rand((n, h, w, ci), generator=g, device="cuda") + 0.5).bfloat16()
    dy = (t.rand((n, h, w, co), generator=g, device="cuda") + 0.5).bfloat16()
    ref = t.zeros((co, ci, 3, 3), dtype=t.float64, device="cuda")
    for b in range(0, n, 16):
        xd, d = x[b:b + 16].double(), dy[b:b + 16].double().reshape(-1, co)
        xp = t.nn.functional.pad(t.cat([xd[:, :, -1:], xd, xd[:, :, :1]], 2), (0, 0, 0, 0, 1, 1))
        for i in range(3):
            for j in range(3):
                ref[:, :, i, j] += d.T @ xp[:, i:i + h, j:j + w].reshape(-1, ci)
    dw = t.zeros((co, ci, 3, 3), device="cuda")
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    assert lib.unet_conv3x3_bwd_weight(vp(x), ci, ci, vp(dy), co, co, vp(dw), None, n, h, w, s) == 0
    assert float(((dw.double() - ref).abs() / ref).max()) < 1.6e-5 + 3e-5
