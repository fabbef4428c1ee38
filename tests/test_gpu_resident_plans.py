"""Resident plans of several sizes alive at once.

Contexts and batch groups of one storage form, relaxation and row class share a
kernel instance but differ in their tiles' shared memory. Each of them keeps
stepping after plans with less of it were made, and all of them give the step
kernel's populations bit for bit.
"""
import numpy as np
import pytest

from paper_0708_4182_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0708_4182_gb300 import lbm as L
    L.load()
    return L


def start(lat, nx, ny):
    mask = wl.channel_mask(nx, ny, amp=4, seed=nx)
    rho = 1.5 + np.cos(np.arange(nx))[None, :] * np.ones((ny, 1))
    lat.set_geometry(mask)
    lat.set_rho(np.where(mask, 0.0, rho))


@pytest.mark.parametrize("sizes", [
    ((128, 64), (301, 67)),      # 34528 and 23504 bytes of the same instance
    ((1024, 128), (1024, 280)),  # 43784 and 40688
    ((1024, 512), (640, 400)),   # 68192 and 67184
    ((2048, 256), (8192, 40)),   # 104864 and 68192
])
def test_two_lattices_stepped_in_turn(lbm, sizes):
    p = dict(wl.PAPER, f_elec=0.1, body_fx=1e-5, storage=lbm.LBM_FP32_DEV)
    lats = [lbm.Lattice(nx, ny, **p) for nx, ny in sizes]
    refs = [lbm.Lattice(nx, ny, layout=lbm.LBM_LAYOUT_SINGLE, **p) for nx, ny in sizes]
    for (nx, ny), a, b in zip(sizes, lats, refs):
        start(a, nx, ny)
        start(b, nx, ny)
    for n in (9, 12):
        for lat in lats:
            lat.step(n)
    for a, b in zip(lats, refs):
        b.step(21)
        assert np.array_equal(a.populations(), b.populations())


@pytest.mark.parametrize("tau,sizes", [
    (0.9, ((489, 90), (683, 256), (640, 102))),   # groups of 39104 and 37544 bytes
    (0.9, ((514, 297), (575, 171), (429, 188))),  # 48296 and 45240
    (0.9, ((501, 13), (614, 369), (1075, 101))),  # 54440 and 46800
    (1.0, ((1011, 132), (773, 554))),             # 101504 and 82784
])
def test_batch_of_several_groups(lbm, tau, sizes):
    p = dict(wl.PAPER, tau=tau, f_elec=0.1, body_fx=1e-5, storage=lbm.LBM_FP32_DEV)
    b = lbm.Batch([dict(nx=nx, ny=ny, **p) for nx, ny in sizes])
    refs = [lbm.Lattice(nx, ny, layout=lbm.LBM_LAYOUT_SINGLE, **p) for nx, ny in sizes]
    for (nx, ny), d, r in zip(sizes, b.domains, refs):
        start(d, nx, ny)
        start(r, nx, ny)
    for n in (60, 51):
        b.step(n)
    for d, r in zip(b.domains, refs):
        r.step(111)
        assert np.array_equal(d.populations(), r.populations())
