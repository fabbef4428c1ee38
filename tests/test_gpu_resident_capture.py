"""A captured even number of steps stays valid between calls that step an even
number of times: the buffer that holds the state after n steps depends on the
parity of n alone, however the steps were run."""
import numpy as np
import pytest

from paper_0708_4182_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    # nx, ny, storage, tau, even step counts between the replays
    (1, 1, 0, 1.0, (2, 4)), (40, 30, 1, 0.9, (2, 4, 6)), (128, 64, 0, 1.0, (2, 4, 8, 1026)),
    (301, 67, 2, 1.0, (2, 10)), (520, 90, 1, 1.0, (4, 34)), (1024, 256, 3, 1.0, (2, 6)), (1024, 512, 0, 1.0, (2, 12)),
]


@pytest.mark.parametrize("nx,ny,storage,tau,counts", CASES)
def test_captured_steps_between_calls(nx, ny, storage, tau, counts):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import lbm
    mask = wl.channel_mask(nx, ny, amp=min(4, (ny - 3) // 2), seed=1) if ny >= 5 else np.zeros((ny, nx), np.uint8)
    if storage >= 2 and nx % 8:
        nx = nx // 8 * 8
        mask = np.ascontiguousarray(mask[:, :nx])
    rho = np.where(mask, 0.0, 1.5 + 0.1 * np.cos(np.arange(nx))[None, :] * np.ones((ny, 1)))
    p = dict(wl.PAPER, tau=tau, f_elec=0.1, body_fx=1e-5, storage=storage)
    st = torch.cuda.Stream()
    lat = lbm.Lattice(nx, ny, stream=st, **p)
    ref = lbm.Lattice(nx, ny, layout=lbm.LBM_LAYOUT_SINGLE, **p)
    for x in (lat, ref):
        x.set_geometry(mask)
        x.set_rho(rho)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        lat.step(2)
    total = 0
    for n in counts:
        lat.step(n)
        with torch.cuda.stream(st):
            g.replay()
        total += n + 2
    ref.step(total)
    assert np.array_equal(lat.populations(), ref.populations())
