"""Updates after a persistent batch whose barrier wait ran out: the maps and the
batch carry nothing of it into the next update."""
import numpy as np
import pytest

import synth
from tests import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BASE = dict(resolution=0.04, noise_a0=0.005, noise_a2=0.002, mahalanobis_k=2.5, outlier_variance=1e-4, ray_step=0.04)
# two maps of the aborted update, and one with the drift compensation, beside
# which the same batch object runs as a kernel sequence
MAPS = [dict(width=90, height=70, wall_num_thresh=3), dict(width=130, height=61), dict(width=40, height=40, flags=1,
                                                                                      drift_flatness=0.9)]


@pytest.fixture(scope="module")
def em():
    from paper_2204_12876_gb300 import build
    build.build()
    from paper_2204_12876_gb300 import em as mod
    return mod


def prior(m, j):
    parity.prior_to_gpu(m, synth.random_prior(seed=40 + j, width=MAPS[j]["width"], height=MAPS[j]["height"], t_now=5,
                                              with_normals=j == 2))


@pytest.mark.parametrize("graph", [False, True])
def test_update_after_a_wait_that_ran_out(em, monkeypatch, graph):
    """No time to wait: the blocks that reach the first barrier before the last one
    leave there, the last one fuses what it can reach and leaves at the second.
    More points than the resident warps take at first, so the work counter is in
    use.  Afterwards the maps, put back to their prior, update through the same
    batch and through em_update as maps that never saw the aborted update."""
    clouds = []
    for j, P in enumerate(MAPS):
        pts, pose = synth.scattered_cloud(50 + j, 3000 if j == 2 else 170_000, 0.5 * P["width"] * 0.04, nan_frac=0.02)
        clouds.append((torch.from_numpy(pts).cuda(), pose))
    monkeypatch.setenv("EM_PERSIST_WAIT_US", "0")
    caps = dict(max_maps=3, max_clouds=3, max_points=400_000, max_cells=130 * 70, graph=graph, persistent=True)
    hurried = em.Batch(**caps)
    monkeypatch.delenv("EM_PERSIST_WAIT_US")
    sound = em.Batch(**caps)
    got = []
    for batch in (hurried, sound):
        maps = [em.Map(em.Params(**BASE, **P)) for P in MAPS]
        for j, m in enumerate(maps):
            prior(m, j)
        if batch is hurried:
            batch.update([(maps[j], *clouds[j]) for j in (0, 1)])
            for j in (0, 1):
                with pytest.raises(em.EMError) as e:
                    maps[j].sync()
                assert e.value.code == em.EM_ERR_TIMEOUT
                maps[j].sync()  # reported once
                prior(maps[j], j)
        before = [m.stats() for m in maps]
        batch.update([(m, *c) for m, c in zip(maps, clouds)])
        maps[0].update(*clouds[0])
        maps[1].shift(5, -3)
        sound.update([(maps[j], *clouds[j]) for j in (0, 1)])
        for m in maps:
            m.sync()
        after = [m.stats() for m in maps]
        got.append(([m.state() for m in maps], [{k: a[k] - b[k] for k in a} for a, b in zip(after, before)]))
    (sa, ta), (sb, tb) = got
    for a, b in zip(sa, sb):
        for k in a:
            assert np.array_equal(a[k], b[k], equal_nan=True), k
    for a, b in zip(ta, tb):
        a.pop("drift_last"), b.pop("drift_last")
        assert a == b
    assert tb[0]["cells_cleared"] > 0 and tb[0]["points_wall"] > 0
    hurried.close()
    sound.close()
