"""Updates whose maps hold far more cells than the clouds have points."""
import numpy as np
import pytest

import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = 0.04
BASE = dict(resolution=R, noise_a0=0.005, noise_a2=0.002, mahalanobis_k=2.5, outlier_variance=1e-4)


@pytest.fixture(scope="module")
def em():
    from paper_2204_12876_gb300 import build
    build.build()
    from paper_2204_12876_gb300 import em as mod
    return mod


def same(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k], equal_nan=True), k


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("ray", [0.0, R])
def test_sparse_and_dense_batches_equal_separate_updates(em, ray, persistent):
    """Batches of more than 2^20 cells with few points (tile flags), with points for
    every other cell (no flags) and with none at all, in turn over the same maps --
    none of them above 2^20 cells by itself, one with the wall rule, one with the
    overlap clearance: as each map's own updates, bit for bit."""
    shapes = [dict(width=700, height=600, wall_num_thresh=2), dict(width=511, height=513), dict(width=640, height=700,
              overlap_radius=0.5, overlap_dz=0.3), dict(width=90, height=33)]
    assert sum(s["width"] * s["height"] for s in shapes) > 1 << 20
    both = []
    for _ in range(2):
        maps = [em.Map(em.Params(**BASE, ray_step=ray, **s)) for s in shapes]
        for j, m in enumerate(maps):
            parity.prior_to_gpu(m, synth.random_prior(seed=j, width=shapes[j]["width"], height=shapes[j]["height"], t_now=5,
                                                      with_normals=False))
            m.shift(7 * j, -3)
        both.append(maps)
    batch = em.Batch(max_maps=4, max_clouds=8, max_points=700_000, max_cells=448_000, persistent=persistent)
    for k, n in enumerate((3000, 170_000, 3000, 0, 500)):
        clouds = []
        for j in range(len(shapes)):
            pts, pose = synth.scattered_cloud(100 * k + j, max(n, 1), 2.0 if n < 10_000 else 14.0, nan_frac=0.02)
            clouds.append((torch.from_numpy(pts[:n]).cuda(), pose))
        batch.update([(m, *c) for m, c in zip(both[0], clouds)])
        for m, c in zip(both[1], clouds):
            m.update(*c)
        for a, b in zip(*both):
            a.sync()
            same(a.state(), b.state())
            assert a.stats() == b.stats()
    if ray:
        assert both[0][1].stats()["cells_cleared"] > 0
    batch.close()


LARGE = [  # beyond 2^19 cells
    dict(width=1000, height=530, ray_step=R),
    dict(width=730, height=729, ray_step=0.0, wall_num_thresh=2, time_variance=1e-6),
    dict(width=600, height=900, ray_step=R, wall_num_thresh=1, flags=1 | 32, cleanup_normal_thresh=0.2,
         drift_flatness=0.9, overlap_radius=0.6, overlap_dz=0.3, excl_b=0.3, excl_c=0.5, excl_theta=0.6, excl_d=1.5),
]


def large_map(em, extra, seed, reserve):
    m = em.Map(em.Params(**{**BASE, **extra}))
    if reserve:
        m.reserve(reserve)
    parity.prior_to_gpu(m, synth.random_prior(seed=seed, width=extra["width"], height=extra["height"], t_now=5))
    m.shift(11, -23)
    return m


@pytest.mark.parametrize("extra", LARGE)
def test_table_of_sums_equals_a_sum_per_cell(em, extra):
    """Maps beyond 2^19 cells keep the sums of the cells the points fall into in a
    table sized for the points; a map reserved for as many points as it has cells
    keeps a sum per cell.  The same updates -- growing, empty, all points in one
    cell, twice the cells of the last -- leave the same map and counters, bit for bit."""
    cells = extra["width"] * extra["height"]
    table, flat = large_map(em, extra, 3, 0), large_map(em, extra, 3, cells)
    assert flat.info()["device_bytes"] > table.info()["device_bytes"] + 30 * cells
    for k, (n, half) in enumerate([(1, 1.0), (4000, 0.5), (40_000, 9.0), (0, 1.0), (33_000, 0.015), (90_000, 15.0)]):
        pts, pose = synth.scattered_cloud(60 + k, max(n, 1), half, nan_frac=0.01)
        d = torch.from_numpy(pts[:n]).cuda()
        for m in (table, flat):
            m.update(d, pose)
            m.sync()
        same(table.state(), flat.state())
        assert table.stats() == flat.stats()
    assert table.stats()["cells_updated"] > 50_000
    if extra["ray_step"]:
        assert table.stats()["cells_cleared"] > 0
    assert table.info()["device_bytes"] < flat.info()["device_bytes"]


@pytest.mark.parametrize("graph, persistent", [(False, False), (True, False), (True, True)])
def test_batches_of_large_and_small_maps(em, graph, persistent):
    """A batch keeps one table for all its maps beyond 2^19 cells, beside the small
    maps' own sums: as each map's own updates, bit for bit."""
    shapes = [LARGE[0], dict(width=90, height=70, ray_step=R), LARGE[1], dict(width=40, height=33, ray_step=R, wall_num_thresh=2)]
    batched, alone = ([large_map(em, s, 10 + j, 0) for j, s in enumerate(shapes)] for _ in range(2))
    batch = em.Batch(max_maps=4, max_clouds=8, max_points=200_000, max_cells=540_000, graph=graph, persistent=persistent)
    for k in range(3):
        clouds = []
        for j, s in enumerate(shapes):
            n = (30_000, 200, 50_000, 70_000)[(j + k) % 4]
            pts, pose = synth.scattered_cloud(20 * k + j, n, (8.0, 1.0)[j % 2], nan_frac=0.01)
            clouds.append((torch.from_numpy(pts).cuda(), pose))
        batch.update([(m, *c) for m, c in zip(batched, clouds)])
        for m, c in zip(alone, clouds):
            m.update(*c)
        batch.update([(batched[0], *clouds[0])])  # one map: its own sums, when it has room, else the batch's
        alone[0].update(*clouds[0])
        for a, b in zip(batched, alone):
            a.sync()
            same(a.state(), b.state())
            assert a.stats() == b.stats()
    batch.close()


def test_persistent_wait_that_ran_out_with_large_maps(em, monkeypatch):
    """The table, too, carries nothing of an update that stopped half way."""
    monkeypatch.setenv("EM_PERSIST_WAIT_US", "0")
    caps = dict(max_maps=2, max_clouds=2, max_points=400_000, max_cells=540_000, persistent=True)
    hurried = em.Batch(**caps)
    pts, pose = synth.scattered_cloud(5, 200_000, 9.0, nan_frac=0.02)
    p = torch.from_numpy(pts).cuda()
    drift = dict(width=40, height=40, flags=1, drift_flatness=0.9, ray_step=R)  # beside it a batch runs as a sequence
    m, ref, small = (large_map(em, s, 7, 0) for s in (LARGE[0], LARGE[0], drift))
    hurried.update([(m, p, pose)])
    with pytest.raises(em.EMError) as e:
        m.sync()
    assert e.value.code == em.EM_ERR_TIMEOUT
    parity.prior_to_gpu(m, synth.random_prior(seed=7, width=1000, height=530, t_now=5))
    parity.prior_to_gpu(ref, synth.random_prior(seed=7, width=1000, height=530, t_now=5))
    hurried.update([(m, p, pose), (small, p, pose)])
    ref.update(p, pose)
    m.sync()
    same(m.state(), ref.state())
    hurried.close()
