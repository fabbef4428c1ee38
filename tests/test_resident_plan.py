"""The grouping of a batch's domains for resident steps, on the host: every group
keeps to the limits that its launch and the exchange buffer rest on."""
import random

import pytest

STORAGE_RECORDS = {0: 3, 1: 3, 2: 2, 3: 2}


@pytest.fixture(scope="module")
def lbm():
    from paper_0708_4182_gb300 import build
    try:
        build.build()
    except RuntimeError as e:
        pytest.skip(f"nvcc unavailable: {e}")
    from paper_0708_4182_gb300 import lbm as L
    return L


def specs(rng, storage, tau):
    out = []
    for _ in range(rng.choice([1, 1, 2, 3, 8, 40])):
        nx, ny = (int(round(2 ** rng.uniform(3, 11))) for _ in range(2))
        if storage >= 2:
            nx = max(8, nx // 8 * 8)
        out.append(dict(nx=nx, ny=ny, storage=storage, tau=tau))
    return out


@pytest.mark.parametrize("edge_nodes", [0, 100000, 30000, 4000])
@pytest.mark.parametrize("storage,tau", [(0, 1.0), (1, 0.9), (2, 1.0), (3, 0.9)])
def test_groups_keep_to_the_limits(lbm, storage, tau, edge_nodes):
    rng = random.Random(storage * 10 + edge_nodes)
    planned = 0
    for _ in range(300):
        sp = specs(rng, storage, tau)
        groups = lbm.lbm_batch_resident_plan(sp, edge_nodes)
        planned += bool(groups)
        if groups:
            assert sum(g["domains"] for g in groups) == len(sp)
        for g in groups:
            assert g["ctas"] * g["edge_nodes"] <= (edge_nodes or 1 << 18)
            per_sm = -(-g["ctas"] // 152)
            assert per_sm * (g["smem"] + 1024) <= 228 * 1024 and g["smem"] <= 227 * 1024
            assert g["threads"] % 32 == 0 and per_sm * g["threads"] <= 2048
            assert g["interval"] in (1, 2, 4)
    assert planned > (20 if edge_nodes == 4000 else 80)


def test_forced_layouts_are_not_grouped(lbm):
    sp = [dict(nx=256, ny=64), dict(nx=40, ny=30)]
    assert len(lbm.lbm_batch_resident_plan(sp)) == 1
    for more in (dict(layout=1), dict(layout=2), dict(tile_rows=8)):
        assert lbm.lbm_batch_resident_plan([sp[0], dict(sp[1], **more)]) == []
    with pytest.raises(lbm.LbmError):
        lbm.lbm_batch_resident_plan([dict(nx=0, ny=5)])
    with pytest.raises(lbm.LbmError):
        lbm.lbm_batch_resident_plan([dict(nx=64, ny=5), dict(nx=64, ny=5, storage=1)])


@pytest.mark.parametrize("storage", [0, 3])
def test_workspace_without_resident_steps(lbm, storage):
    """A batch with a forced layout or height carries no exchange buffer (16 bytes
    per record, two buffers of 2^18 nodes) and no CTA table."""
    sp = [dict(nx=256, ny=64, storage=storage), dict(nx=40, ny=30, storage=storage)]

    def size(**more):
        arr = (lbm.lbm_params * 2)(*[lbm.make_params(**{**sp[0], **more}), lbm.make_params(**sp[1])])
        return lbm._batch_lib().lbm_batch_workspace_bytes(arr, 2)

    exchange = 2 * 16 * STORAGE_RECORDS[storage] << 18
    for more in (dict(layout=1), dict(layout=2), dict(tile_rows=8)):
        assert size() - size(**more) >= exchange
