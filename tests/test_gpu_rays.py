"""The ray march's chunk test and its order of work (k_points, k_refresh).

Against the FP64 oracle (tolerances and marginal bands of tests/parity.py): map
sides around the 8 x 8 blocks of the coarse grid and its rim, sensors outside
the map, steps from half a cell to twenty.  Bit for bit: the points of one
large cloud in a sensor's order (one part) and shuffled (parts with refreshed
thresholds between them)."""
import numpy as np
import pytest

import oracle
import synth
from . import parity

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = 0.04


@pytest.fixture(scope="module")
def em():
    from paper_2204_12876_gb300 import build
    build.build()
    from paper_2204_12876_gb300 import em as mod
    return mod


@pytest.mark.parametrize("W, H", [(1, 1), (7, 9), (8, 8), (33, 65), (120, 17)])
@pytest.mark.parametrize("step", [0.02, 0.04, 0.13, 0.8])
@pytest.mark.parametrize("outside", [False, True])
def test_small_maps_steps_and_sensors(em, W, H, step, outside):
    P = dict(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002, var_min=1e-8, mahalanobis_k=2.5,
             outlier_variance=1e-4, ray_step=step)
    rng = np.random.default_rng(W * 100 + H)
    prior = synth.random_prior(seed=W + H, width=W, height=H, t_now=5, obstacle_frac=0.3, with_normals=False)
    half = np.array([W, H]) * R / 2
    t = np.array([half[0] + 0.7, -half[1] - 0.4, 0.6]) if outside else np.array([0.0, 0.0, 0.5])
    n = 3000
    xy = rng.uniform(-1.5, 1.5, (n, 2)) * (half + 0.2)
    pw = np.concatenate([xy, rng.normal(0.0, 0.1, (n, 1))], axis=1)
    pts, pose = (pw - t).astype(np.float32), synth.pose_matrix(np.eye(3), t)
    om = oracle.OracleMap(parity.oracle_params(P))
    parity.prior_to_oracle(om, prior)
    prior_valid = np.isfinite(om.state()["var"])
    tr = om.update((pts, pose), trace=True, unit=oracle.FP32_UNIT, abs_band=parity.ABS_BAND)
    m = em.Map(em.Params(**P, flags=em.F_TRACE))
    parity.prior_to_gpu(m, prior)
    m.update(torch.from_numpy(pts).cuda(), pose)
    # (a handful of cells: no bound on the share of marginal ones)
    parity.compare_update(tr, om.state(), m.state(), m.trace(n), check_stencils=(), prior_valid=prior_valid,
                          max_excluded=1.0)
    m.close()


@pytest.mark.parametrize("upper", [False, True])
@pytest.mark.parametrize("batched", [False, True])
def test_parts_equal_one_part(em, upper, batched):
    side, n = 300, 1_100_000  # beyond the size from which scattered points go in parts
    pts, pose = synth.scattered_cloud(91, n, 0.5 * side * R * 1.05, nan_frac=0.01)
    az = np.floor(np.nan_to_num(np.arctan2(pts[:, 1], pts[:, 0])) * 115).astype(np.int64)
    order = np.lexsort((np.nan_to_num(np.linalg.norm(pts, axis=1)), az))  # along the rays of a turning sensor
    prior = synth.random_prior(seed=92, width=side, height=side, t_now=5, with_normals=False)
    got = []
    for cloud in (pts, np.ascontiguousarray(pts[order])):
        m = em.Map(em.Params(width=side, height=side, resolution=R, noise_a0=0.005, noise_a2=0.002, mahalanobis_k=2.5,
                             outlier_variance=1e-4, ray_step=R, flags=em.F_UPPER if upper else 0))
        parity.prior_to_gpu(m, prior)
        p = torch.from_numpy(cloud).cuda()
        if batched:
            b = em.Batch(max_maps=1, max_clouds=1, max_points=n, max_cells=side * side)
            for _ in range(2):
                b.update([(m, p, pose)])
            torch.cuda.synchronize()
            b.close()
        else:
            for _ in range(2):
                m.update(p, pose)
        got.append((m.state(), m.stats()))
        m.close()
    (a, sa), (c, sc) = got
    for k in ("h", "var", "t_last") + (("upper",) if upper else ()):
        assert np.array_equal(a[k], c[k], equal_nan=True), k
    assert sa == sc and sa["cells_cleared"] > 0 and sa["ray_samples"] > 0


@pytest.mark.parametrize("graph, persistent", [(False, False), (True, False), (True, True)])
@pytest.mark.parametrize("upper", [False, True])
def test_batches_in_parts_equal_separate_updates(em, upper, graph, persistent):
    """Two maps of different sizes whose clouds together reach the size from which
    scattered points go in parts, each below it by itself: the batch, in parts with
    refreshed thresholds, leaves what the maps' own updates leave, bit for bit --
    with the wall rule, the time variance, the Eq. 4 guard, the upper-bound layer."""
    specs = [dict(width=300, height=290, cleanup_normal_thresh=0.3, flags=em.F_NORMALS | (em.F_UPPER if upper else 0)),
             dict(width=211, height=333, wall_num_thresh=3, time_variance=1e-6, ray_step=0.06)]
    counts = (620_000, 480_000)
    assert sum(counts) > 1 << 20 > max(counts)
    base = dict(resolution=R, noise_a0=0.005, noise_a2=0.002, mahalanobis_k=2.5, outlier_variance=1e-4, ray_step=R)
    both = []
    for _ in range(2):
        maps = [em.Map(em.Params(**{**base, **s})) for s in specs]
        for j, m in enumerate(maps):
            parity.prior_to_gpu(m, synth.random_prior(seed=95 + j, width=specs[j]["width"], height=specs[j]["height"],
                                                      t_now=5, with_normals=j == 0))
            m.shift(17, -40 * j)
        both.append(maps)
    b = em.Batch(max_maps=2, max_clouds=2, max_points=sum(counts), max_cells=300 * 300, graph=graph, persistent=persistent)
    for k in range(2):
        clouds = []
        for j, n in enumerate(counts):
            pts, pose = synth.scattered_cloud(97 + 2 * k + j, n, 6.3, nan_frac=0.01)
            clouds.append((torch.from_numpy(pts).cuda(), pose))
        b.update([(m, *c) for m, c in zip(both[0], clouds)])
        for m, c in zip(both[1], clouds):
            m.update(*c)
        for x, y in zip(*both):
            x.sync()
            s, t = x.state(), y.state()
            for key in s:
                assert np.array_equal(s[key], t[key], equal_nan=True), (k, key)
            assert x.stats() == y.stats()
    assert both[0][0].stats()["cells_cleared"] > 0 and both[0][1].stats()["points_wall"] > 0
    b.close()


@pytest.mark.parametrize("W, H", [(1, 1), (7, 9), (8, 8), (9, 1)])
def test_cells_of_tiny_maps_are_compared(em, W, H):
    """Few points, so that few cells are marginal: over several scenes most cells of
    maps of one and a few cells agree with the oracle, none of them excluded."""
    compared = valid = 0
    for seed in range(24):
        rng = np.random.default_rng(seed)
        P = dict(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002, var_min=1e-8, mahalanobis_k=2.5,
                 outlier_variance=1e-4, ray_step=(0.02, 0.04, 0.13)[seed % 3])
        prior = synth.random_prior(seed=seed, width=W, height=H, t_now=5, obstacle_frac=0.3, with_normals=False)
        half, t = np.array([W, H]) * R / 2, np.array([0.3 * (seed % 2), -0.2 * (seed % 2), 0.5])
        pw = np.concatenate([rng.uniform(-1.5, 1.5, (40, 2)) * (half + 0.1), rng.normal(0.0, 0.1, (40, 1))], axis=1)
        pts, pose = (pw - t).astype(np.float32), synth.pose_matrix(np.eye(3), t)
        om = oracle.OracleMap(parity.oracle_params(P))
        parity.prior_to_oracle(om, prior)
        prior_valid = np.isfinite(om.state()["var"])
        tr = om.update((pts, pose), trace=True, unit=oracle.FP32_UNIT, abs_band=parity.ABS_BAND)
        m = em.Map(em.Params(**P, flags=em.F_TRACE))
        parity.prior_to_gpu(m, prior)
        m.update(torch.from_numpy(pts).cuda(), pose)
        cmp = parity.compare_update(tr, om.state(), m.state(), m.trace(40), check_stencils=(), prior_valid=prior_valid,
                                    max_excluded=1.0)
        m.close()
        compared += cmp.notes["cells_compared"]
        valid += int(np.isfinite(om.state()["var"]).sum())
    assert valid > 0 and compared > valid / 2, (compared, valid)
