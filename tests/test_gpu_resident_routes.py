"""Which calls run in the resident kernel: the comparisons with the step kernel
mean nothing where both sides take the same way."""
import numpy as np
import pytest
from test_gpu_resident import CASES, domain

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


def ready(lbm, nx, ny, **more):
    p = dict(wl.PAPER, f_elec=0.1, body_fx=1e-5, **more)
    lat = lbm.Lattice(nx, ny, **p)
    mask, rho = domain(nx, ny, True, 1)
    lat.set_geometry(mask)
    lat.set_rho(np.where(mask, 0.0, 1.5 + 0 * rho))
    return lat


@pytest.mark.parametrize("nx,ny,walls,storage,tau", CASES)
def test_compared_domains_are_resident(lbm, nx, ny, walls, storage, tau):
    lat = ready(lbm, nx, ny, storage=storage, tau=tau)
    lat.step(9)
    assert lat.resident_launches == 1
    lat.step(1)
    assert lat.resident_launches == 1  # a single step is a launch of its own


@pytest.mark.parametrize("more", [
    dict(layout=1), dict(layout=2), dict(tile_rows=8), dict(obs_every=1), dict(nx=1024, ny=900), dict(nx=1024, ny=512, tau=0.9),
])
def test_other_calls_are_not(lbm, more):
    more = dict(more)
    lat = ready(lbm, more.pop("nx", 128), more.pop("ny", 64), **more)
    lat.step(40)
    lat.observables()
    assert lat.resident_launches == 0


@pytest.mark.parametrize("nx,ny,storage,two", [
    (128, 64, 0, 1), (1024, 290, 0, 1), (90, 5000, 0, 1), (1024, 512, 0, 0), (2048, 256, 0, 0), (1024, 512, 1, 1),
    (1024, 580, 1, 0), (1024, 512, 2, 1),
])
def test_two_steps_of_large_domains_are_not(lbm, nx, ny, storage, two):
    lat = ready(lbm, nx, ny, storage=storage)
    lat.step(2)
    assert lat.resident_launches == two
    lat.step(3)
    assert lat.resident_launches == two + 1


def test_captured_steps_are_not(lbm):
    import torch
    st = torch.cuda.Stream()
    lat = lbm.Lattice(128, 64, stream=st, **wl.PAPER)
    mask, _ = domain(128, 64, True, 1)
    lat.set_geometry(mask)
    lat.set_rho(np.where(mask, 0.0, 1.5))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        lat.step(6)
    assert lat.resident_launches == 0
    lat.step(6)
    assert lat.resident_launches == 1


@pytest.mark.parametrize("tau,sizes,groups", [
    (1.0, ((256, 64), (40, 30), (320, 200), (64, 4), (8, 100), (264, 61), (512, 256)), 1),
    (0.9, ((514, 297), (575, 171), (429, 188)), 2), (1.0, ((1011, 132), (773, 554)), 2),
])
def test_batches(lbm, tau, sizes, groups):
    p = dict(wl.PAPER, tau=tau, storage=lbm.LBM_FP32_DEV)
    for more, resident in ((dict(), True), (dict(layout=lbm.LBM_LAYOUT_SINGLE), False), (dict(tile_rows=16), False)):
        b = lbm.Batch([dict(nx=nx, ny=ny, **p, **more) for nx, ny in sizes])
        for (nx, ny), d in zip(sizes, b.domains):
            mask, _ = domain(nx, ny, True, nx)
            d.set_geometry(mask)
            d.set_rho(np.where(mask, 0.0, 1.5))
        b.step(50)
        b.observables()
        assert (b.resident_groups, b.resident_launches) == ((groups, groups) if resident else (0, 0))


def test_larger_plans_stay_resident(lbm):
    lats = [ready(lbm, nx, ny, storage=lbm.LBM_FP32_DEV) for nx, ny in ((2048, 256), (1024, 512), (640, 400), (128, 64), (301, 67))]
    for lat in lats:
        lat.step(20)
        lat.observables()
        assert lat.resident_launches == 1


@pytest.mark.parametrize("nx,ny,storage", [(128, 64, 0), (1024, 128, 1), (1024, 512, 0), (2048, 256, 1), (1024, 580, 2)])
def test_a_launch_holds_the_gpu_for_some_milliseconds(lbm, nx, ny, storage):
    """Three by the plan's estimate, which may be off by half."""
    import torch
    lat = ready(lbm, nx, ny, storage=storage)
    lat.step(1024)
    before, start, end = lat.resident_launches, *(torch.cuda.Event(enable_timing=True) for _ in range(2))
    start.record()
    lat.step(2048)
    end.record()
    torch.cuda.synchronize()
    assert start.elapsed_time(end) / (lat.resident_launches - before) < 4.5


def test_a_group_holds_the_gpu_for_some_milliseconds(lbm):
    import torch
    p = dict(wl.PAPER, storage=lbm.LBM_FP32_DEV)
    b = lbm.Batch([dict(nx=256, ny=64, **p) for _ in range(64)])
    for d in b.domains:
        mask, _ = domain(256, 64, True, 1)
        d.set_geometry(mask)
        d.set_rho(np.where(mask, 0.0, 1.5))
    b.step(500)
    before, start, end = b.resident_launches, *(torch.cuda.Event(enable_timing=True) for _ in range(2))
    start.record()
    b.step(1000)
    end.record()
    torch.cuda.synchronize()
    assert start.elapsed_time(end) / (b.resident_launches - before) < 4.5
