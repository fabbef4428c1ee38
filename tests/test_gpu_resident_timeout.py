"""The resident steps' bounded wait, without a fault: the self-test polls records
that nothing writes (after the step kernel's own wait), both waits give up, and
the context steps on."""
import time

import numpy as np
import pytest

from paper_0708_4182_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_record_wait_gives_up():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import lbm
    lats = []
    for lay in (lbm.LBM_LAYOUT_AUTO, lbm.LBM_LAYOUT_SINGLE):
        lat = lbm.Lattice(301, 67, layout=lay, **wl.PAPER)
        mask = wl.channel_mask(301, 67, amp=4, seed=1)
        lat.set_geometry(mask)
        lat.set_rho(np.where(mask, 0.0, 1.5))
        lat.step(10)
        lats.append(lat)
    t0 = time.perf_counter()
    assert lbm.lbm_selftest_timeout(lats[0].ctx) == lbm.LBM_ETIMEOUT
    # 2^18 and 2^20 polls: well over a millisecond each, and an end
    assert 0.01 < time.perf_counter() - t0 < 20.0
    for lat in lats:
        lat.step(10)
    assert lats[0].resident_launches == 2
    assert np.array_equal(lats[0].populations(), lats[1].populations())
