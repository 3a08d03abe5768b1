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
