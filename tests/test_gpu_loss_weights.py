"""The weighted loss counts exactly the given elements: an infinite class
weight gives an infinite loss, whatever the element count leaves over."""
import ctypes
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,c,hw", [(1, 1, 5), (2, 3, 1000), (3, 3, 4097)])
def test_infinite_weight(n, c, hw):
    import torch as t
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import surrogate
    lib = surrogate.load_unet()
    vp = lambda a: ctypes.c_void_p(a.data_ptr())  # noqa: E731
    p, q = t.ones((n, c, hw), device="cuda"), t.zeros((n, c, hw), device="cuda")
    wc = t.full((c,), math.inf, device="cuda")
    grad, loss = t.empty_like(p), t.zeros(1, dtype=t.float64, device="cuda")
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    assert lib.unet_mse(vp(p), vp(q), vp(wc), c, hw, n * c * hw, vp(grad), vp(loss), s) == 0
    assert float(loss) == math.inf
    assert bool((grad == math.inf).all())
