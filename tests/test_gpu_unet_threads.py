"""Convolutions of several widths called from several host threads at once,
each on its own stream: the calls of one kernel instance need different amounts
of shared memory, and none of them may take another's away."""
import ctypes
import threading

import pytest

pytestmark = pytest.mark.gpu


def test_convolutions_from_threads():
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import surrogate
    lib = surrogate.load_unet()
    vp = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    ci, co, n, h = 64, 32, 1, 4
    wt = t.randn((co, ci, 3, 3), device="cuda") * 0.05
    pk = t.empty(int(lib.unet_conv_pack_elems(co, ci, 0)), dtype=t.bfloat16, device="cuda")
    s0 = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    assert lib.unet_conv_pack(vp(wt), co, ci, 0, vp(pk), s0) == 0
    widths = (32, 224, 96, 160)
    data = []
    for w in widths:
        x = t.randn((n, h, w, ci), device="cuda").bfloat16()
        want = t.empty((n, h, w, co), dtype=t.bfloat16, device="cuda")
        assert lib.unet_conv3x3(vp(x), ci, ci, vp(pk), None, vp(want), co, co, n, h, w, 0, s0) == 0
        data.append((w, x, want, t.empty_like(want), t.cuda.Stream()))
    t.cuda.synchronize()
    failed = []

    def work(w, x, want, y, st):
        s = ctypes.c_void_p(st.cuda_stream)
        for _ in range(2000):
            rc = lib.unet_conv3x3(vp(x), ci, ci, vp(pk), None, vp(y), co, co, n, h, w, 0, s)
            if rc:
                failed.append((w, rc))
                return

    threads = [threading.Thread(target=work, args=d) for d in data]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    t.cuda.synchronize()
    assert not failed
    for w, _, want, y, _ in data:
        assert t.equal(y, want), w
