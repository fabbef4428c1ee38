"""Weight gradients of two shapes on two streams at once. Their CTAs fit on one
SM by shared memory (78,848 and about 148,100 bytes) but not by tensor memory
(256 and 512 columns), and both shapes are small enough to run in clusters:
no CTA may keep its columns while it waits for its cluster."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w", [32, 16])
def test_two_instances_at_once(w):
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import surrogate
    lib = surrogate.load_unet()
    vp = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    runs = []
    for n, ci, co, h, wd in ((4, 16, 32, 16, w), (4, 32, 32, 16, 64)):
        x = t.randn((n, h, wd, ci), device="cuda").bfloat16()
        dy = t.randn((n, h, wd, co), device="cuda").bfloat16()
        alone = t.zeros((co, ci, 3, 3), device="cuda")
        s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
        assert lib.unet_conv3x3_bwd_weight(vp(x), ci, ci, vp(dy), co, co, vp(alone), None, n, h, wd, s) == 0
        runs.append((n, ci, co, h, wd, x, dy, alone, [t.zeros_like(alone) for _ in range(200)], t.cuda.Stream()))
    t.cuda.synchronize()
    for i in range(200):
        for n, ci, co, h, wd, x, dy, _, dws, st in runs:
            s = ctypes.c_void_p(st.cuda_stream)
            assert lib.unet_conv3x3_bwd_weight(vp(x), ci, ci, vp(dy), co, co, vp(dws[i]), None, n, h, wd, s) == 0
    t.cuda.synchronize()
    for *_, alone, dws, _ in runs:
        # the same sums, up to the order of the FP32 atomics (a few addends)
        for dw in dws:
            assert float(t.linalg.norm(dw - alone) / t.linalg.norm(alone)) < 1e-6
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    assert lib.unet_tc_error(s, 1) == 0
