"""Resident steps (many time steps per launch, the state in shared memory)
against the step kernel.

Domains that fit on the chip take the resident kernel in the automatic
layout; a forced thread layout always takes the step kernel. Both run the same
node arithmetic, so the populations are equal bit for bit whatever the tiling.
The sizes sit at the edges of the tiling: domains smaller than a halo, widths
around multiples of the 30, 26 and 18 columns of a tile, one-tile and many-tile
directions, the largest domains, and step counts that end a round of exchanges
early or span several launches.
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


def domain(nx, ny, walls, seed):
    rng = np.random.default_rng(seed)
    if walls and ny >= 5:
        mask = wl.channel_mask(nx, ny, amp=min(6, (ny - 3) // 2), seed=seed)
        if nx > 40 and ny > 20:
            mask[9:12, nx // 2:nx // 2 + 3] = 1  # an obstacle in the fluid
    else:
        mask = np.zeros((ny, nx), np.uint8)
    rho = np.where(mask, 0.0, 0.3 + 2.4 * rng.random((ny, nx)))
    return mask, rho


CASES = [
    # nx, ny, walls, storage, tau
    (1, 1, False, 0, 1.0), (2, 3, False, 1, 1.0), (7, 5, False, 0, 0.9), (8, 3, False, 2, 1.0),
    (17, 40, True, 0, 1.0), (18, 19, True, 1, 1.0), (26, 27, False, 0, 1.0), (30, 150, True, 1, 0.9),
    (31, 61, True, 0, 1.0), (64, 32, True, 3, 0.9), (61, 300, True, 1, 1.0), (128, 64, True, 0, 0.9),
    (301, 67, True, 0, 1.0), (520, 90, True, 1, 1.0), (1024, 128, True, 3, 1.0), (1023, 257, True, 0, 1.0),
    (1024, 512, True, 1, 1.0), (8192, 40, True, 2, 1.0), (90, 5000, True, 0, 1.0),
]


@pytest.mark.parametrize("nx,ny,walls,storage,tau", CASES)
def test_resident_steps_equal_the_step_kernel(lbm, nx, ny, walls, storage, tau):
    mask, rho = domain(nx, ny, walls, nx + ny)
    # 16-bit states round off faster from random densities: a smoother start
    if storage >= 2:
        rho = np.where(mask, 0.0, 1.5 + 0.1 * np.cos(np.arange(nx))[None, :] * np.ones((ny, 1)))
    p = dict(wl.PAPER, tau=tau, f_elec=0.1, body_fx=1e-5)
    lats = [lbm.Lattice(nx, ny, storage=storage, layout=lay, **p) for lay in (lbm.LBM_LAYOUT_AUTO, lbm.LBM_LAYOUT_SINGLE)]
    for lat in lats:
        lat.set_geometry(mask)
        lat.set_rho(rho)
    for n in (2, 3, 9, 32):
        for lat in lats:
            lat.step(n)
        a, b = (lat.populations() for lat in lats)
        assert np.array_equal(a, b, equal_nan=True), n
    assert lats[0].time == lats[1].time == 46


def test_resident_steps_over_several_launches_and_observed_steps(lbm):
    w = wl.rough_channel(nx=140, ny=50, amp=5, level=9, seed=3)
    obs = []
    pops = []
    for lay in (lbm.LBM_LAYOUT_AUTO, lbm.LBM_LAYOUT_SINGLE):
        lat = lbm.Lattice(w.nx, w.ny, storage=lbm.LBM_FP32_DEV, obs_every=700, layout=lay, **w.params)
        lat.set_geometry(w.mask)
        lat.set_rho(w.rho)
        lat.step(2500)
        obs.append(lat.obs_latest())
        lat.set_rho(w.rho)  # the exchange goes on with the tags of the last run
        lat.step(5)
        pops.append(lat.populations())
    assert obs[0]["step"] == obs[1]["step"] == 2100
    for k in ("mass", "flux_Q", "mom_x", "mom_y", "max_u", "min_rho"):
        assert obs[0][k] == pytest.approx(obs[1][k], rel=1e-12, abs=1e-15), k
    assert np.array_equal(pops[0], pops[1])


@pytest.mark.parametrize("storage,tau", [(0, 1.0), (1, 1.0), (1, 0.9), (3, 1.0)])
def test_resident_batch_equals_domains_stepped_alone(lbm, storage, tau):
    sizes = [(256, 64), (40, 30), (320, 200), (64, 4), (8, 100), (264, 61), (512, 256)]
    p = dict(wl.PAPER, tau=tau, f_elec=0.1, body_fx=1e-5)
    b = lbm.Batch([dict(nx=nx, ny=ny, storage=storage, **p) for nx, ny in sizes])
    alone = []
    for (nx, ny), d in zip(sizes, b.domains):
        mask, _ = domain(nx, ny, True, nx)
        rho = np.where(mask, 0.0, 1.5 + np.cos(np.arange(nx))[None, :] * np.ones((ny, 1)))
        lat = lbm.Lattice(nx, ny, storage=storage, layout=lbm.LBM_LAYOUT_SINGLE, **p)
        for x in (d, lat):
            x.set_geometry(mask)
            x.set_rho(rho)
        alone.append(lat)
    active = [True] * len(sizes)
    for n in (50, 21):  # then without the third domain
        b.set_active(active)
        b.step(n)
        for lat, on in zip(alone, active):
            if on:
                lat.step(n)
        for d, lat in zip(b.domains, alone):
            assert np.array_equal(d.populations(), lat.populations()), (n, d.nx, d.ny)
            assert d.time == lat.time
        active[2] = False


def test_concurrent_streams(lbm):
    """Two domains stepped on two streams at once: each launch holds all its
    CTAs, so the two take turns or share the SMs, and neither waits for the
    other inside a kernel."""
    import torch
    w = wl.rough_channel(nx=1024, ny=128, amp=4, level=5, seed=1)
    ref = lbm.Lattice(w.nx, w.ny, **w.params)
    ref.set_geometry(w.mask)
    ref.set_rho(w.rho)
    ref.step(600)
    want = ref.populations()
    lats = []
    for _ in range(2):
        st = torch.cuda.Stream()
        lat = lbm.Lattice(w.nx, w.ny, stream=st, **w.params)
        lat.set_geometry(w.mask)
        lat.set_rho(w.rho)
        lats.append(lat)
    for _ in range(6):
        for lat in lats:
            lat.step(100)
    for lat in lats:
        assert np.array_equal(lat.populations(), want)
