"""The points' way into their cells (k_points, k_write): runs of equal cells in
consecutive lanes, batches of 32 points across clouds and maps, map sizes
around the kernels' tiles, and weights that vanish in fixed point.

Expected values are the per-cell inverse-variance means in float64 (Eq. 1/2
over an empty map, Section II-C), with the repository's tolerances for the
float32 path: heights 1e-5 m, variances 1e-4 relative."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

R = 0.04
POSE = np.array([1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0.0], np.float32)


@pytest.fixture(scope="module")
def em():
    from paper_2204_12876_gb300 import build
    build.build()
    from paper_2204_12876_gb300 import em as mod
    return mod


def runs_cloud(rng, W, H, n):
    """n points in runs of 1, 2, 31, 32, 33 and 70 points of one cell, well inside their cells."""
    cells = []
    lengths = [1, 2, 31, 32, 33, 70, 5]
    while len(cells) < n:
        cells += [(int(rng.integers(W)), int(rng.integers(H)))] * lengths[len(cells) % len(lengths)]
    c = np.array(cells[:n])
    xy = (c + 0.5 + rng.uniform(-0.3, 0.3, (n, 2)) - np.array([W, H]) / 2) * R
    p = np.concatenate([xy, rng.uniform(-0.8, -0.3, (n, 1))], axis=1).astype(np.float32)
    return p, c


def expected(parts, W, H, a0, a2):
    """Per-cell (h, var) of points over an empty map, float64."""
    sw, swz = np.zeros((H, W)), np.zeros((H, W))
    for p, c in parts:
        p = p.astype(np.float64)
        w = 1.0 / (a0 + a2 * (p * p).sum(axis=1)) ** 2
        np.add.at(sw, (c[:, 1], c[:, 0]), w)
        np.add.at(swz, (c[:, 1], c[:, 0]), w * p[:, 2])
    with np.errstate(invalid="ignore", divide="ignore"):
        return swz / sw, 1.0 / sw


def check(state, parts, W, H, a0=0.005, a2=0.002):
    h, var = expected(parts, W, H, a0, a2)
    hit = np.isfinite(h)
    assert np.array_equal(np.isfinite(state["var"]), hit)
    assert np.all(np.abs(state["h"][hit] - h[hit]) <= 1e-5)
    assert np.all(np.abs(state["var"][hit] / var[hit] - 1.0) <= 1e-4)


@pytest.mark.parametrize("W, H, n", [(1, 1, 1), (1, 1, 100), (31, 33, 31), (32, 32, 33), (33, 31, 1023),
                                     (1025, 1, 2049), (64, 48, 20001)])
@pytest.mark.parametrize("ray", [False, True])
def test_runs_and_map_sizes(em, W, H, n, ray):
    rng = np.random.default_rng(W * 7919 + n)
    m = em.Map(em.Params(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002,
                         ray_step=R if ray else 0.0))
    p, c = runs_cloud(rng, W, H, n)
    m.update(torch.from_numpy(p).cuda(), POSE)
    check(m.state(), [(p, c)], W, H)
    st = m.stats()
    assert st["points_valid"] == st["points_in_map"] == st["points_accepted"] == n and st["points_rejected"] == 0
    assert st["cells_updated"] == len(np.unique(c[:, 1] * W + c[:, 0])) and st["updates"] == 1
    m.close()


@pytest.mark.parametrize("persistent", [False, True])
def test_batches_of_points_across_clouds_and_maps(em, persistent):
    """Clouds of 1 to 97 points: most 32-point batches hold several clouds, many several maps."""
    rng = np.random.default_rng(3)
    sizes = [(20, 13), (1, 1), (40, 40), (7, 90)]
    maps = [em.Map(em.Params(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002, ray_step=R))
            for W, H in sizes]
    pairs, parts = [], [[] for _ in sizes]
    for n in (1, 5, 31, 97, 64, 3, 17):
        for j, (W, H) in enumerate(sizes):
            p, c = runs_cloud(rng, W, H, n)
            parts[j].append((p, c))
            pairs.append((maps[j], torch.from_numpy(p).cuda(), POSE))
    batch = em.Batch(max_maps=4, max_clouds=len(pairs), max_points=4096, max_cells=1600, persistent=persistent)
    batch.update(pairs)
    for j, (W, H) in enumerate(sizes):
        maps[j].sync()
        check(maps[j].state(), parts[j], W, H)
        assert maps[j].stats()["points_accepted"] == sum(len(p) for p, _ in parts[j])
    batch.close()


def test_weights_below_fixed_point(em):
    """A point whose weight is below 2^-44 still counts as accepted: a valid cell
    keeps its height, its variance (to rounding) and gets the update's index."""
    m = em.Map(em.Params(width=2, height=1, resolution=R, noise_a0=1e8))
    h = np.array([[0.25, np.nan]], np.float32)
    var = np.array([[0.01, np.inf]], np.float32)
    m.set_state(h=h, var=var, t_last=np.zeros((1, 2), np.float32), t_now=4)
    p = np.array([[-0.02, 0.0, 1.0]] * 40, np.float32)
    m.update(torch.from_numpy(p).cuda(), POSE)
    s = m.state()
    assert s["h"][0, 0] == np.float32(0.25) and abs(s["var"][0, 0] / 0.01 - 1) < 1e-6
    assert s["t_last"][0, 0] == 5 and s["t_last"][0, 1] == 0
    assert m.stats()["points_accepted"] == 40 and m.stats()["cells_updated"] == 1
    m.close()


def test_updates_under_stream_capture(em):
    """The one-map forms take their descriptor as a kernel parameter, so an update
    captured from a stream replays whole: each replay fuses the cloud again as
    the update index it was captured with."""
    rng = np.random.default_rng(5)
    W, H, n = 40, 33, 5000
    p, _ = runs_cloud(rng, W, H, n)
    d = torch.from_numpy(p).cuda()
    P = em.Params(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002, ray_step=R)
    states = []
    for captured in (False, True):
        m = em.Map(P)
        m.reserve(n)
        h, v = torch.full((H, W), float("nan"), device="cuda"), torch.full((H, W), float("inf"), device="cuda")
        t = torch.zeros((H, W), dtype=torch.int32, device="cuda")
        em.update_noalloc(P, h, v, t, [(d, POSE)], t_now=1)  # (its first call looks up the scratch)
        out = torch.empty(3, H, W, device="cuda")
        torch.cuda.synchronize()

        def step():
            m.update(d, POSE)
            em.update_noalloc(P, h, v, t, [(d, POSE)], t_now=2)
            m.get_layers(em.LAYER_ELEVATION | em.LAYER_VARIANCE | em.LAYER_TIME, out=out)

        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                step()
            for _ in range(2):
                g.replay()
        else:
            for _ in range(2):
                step()
                m.set_state(t_now=0)  # the captured update keeps its index
        torch.cuda.synchronize()
        states.append([x.cpu().numpy() for x in (out, h, v, t)])
        m.close()
    for a, b in zip(*states):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("graph", [False, True])
def test_batch_of_one_map_equals_update(em, graph):
    """A batch that names one map (once, or with several clouds) runs as em_update
    does: same state and counters as Map.update_multi, also beside batches of two."""
    rng = np.random.default_rng(6)
    W, H = 50, 41
    make = lambda: em.Map(em.Params(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002,  # noqa: E731
                                    mahalanobis_k=2.5, outlier_variance=1e-4, ray_step=R))
    clouds = [[torch.from_numpy(runs_cloud(rng, W, H, n)[0]).cuda() for n in ns] for ns in ((3000,), (700, 5, 900), (64,))]
    ref, m, other = make(), make(), make()
    batch = em.Batch(max_maps=2, max_clouds=8, max_points=8192, max_cells=W * H, graph=graph)
    for k, cs in enumerate(clouds):
        ref.update_multi([(c, POSE) for c in cs])
        pairs = [(m, c, POSE) for c in cs]
        batch.update(pairs + [(other, cs[0], POSE)] if k == 1 else pairs)
    a, b = ref.state(), m.state()
    for k in ("h", "var", "t_last"):
        assert np.array_equal(a[k], b[k], equal_nan=True), k
    assert ref.stats() == m.stats() and m.info()["t_now"] == 3
    with pytest.raises(em.EMError) as e:  # the batch's capacities hold for one map too
        batch.update([(m, torch.zeros(9000, 3, device="cuda"), POSE)])
    assert e.value.code == em.EM_ERR_CAPACITY and m.info()["t_now"] == 3
    batch.close()


@pytest.mark.parametrize("extra", [dict(), dict(ray_step=0.0), dict(wall_num_thresh=2, time_variance=1e-6),
                                   dict(drift_flatness=0.9, cleanup_normal_thresh=0.1, overlap_radius=0.5,
                                        overlap_dz=0.2, excl_b=0.2, excl_c=0.3, excl_theta=0.5, excl_d=1.0,
                                        flags=1 | 4 | 8 | 32)])
def test_uploaded_descriptor_equals_parameter(em, extra):
    """Updates of more than 8 clouds upload their descriptor, the others pass it as
    a kernel parameter: the same points as 1, 3 and 12 clouds -- strides 3 and 4,
    rows off a 16-byte boundary, ragged and empty clouds -- leave the same map and
    counters, over two updates with a shift between them."""
    import synth
    W, H, n = 70, 53, 9000
    pts, pose = synth.scattered_cloud(8, n, 1.3, nan_frac=0.02)
    prior = synth.random_prior(seed=9, width=W, height=H, t_now=5)
    P = dict(dict(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002, mahalanobis_k=2.5,
                  outlier_variance=1e-4, ray_step=R), **extra)
    got = []
    for parts in (1, 3, 12):
        cuts = np.sort(np.random.default_rng(parts).integers(0, n + 1, parts - 1))
        if parts > 2:
            cuts[1] = cuts[0]  # an empty cloud
        clouds = []
        for k, c in enumerate(np.split(pts, cuts)):
            c = np.concatenate([c, np.zeros((len(c), 1), np.float32)], axis=1) if k % 3 == 1 else c
            flat = torch.zeros(c.size + 1, device="cuda")[1:] if k % 2 else torch.zeros(c.size, device="cuda")
            flat.copy_(torch.from_numpy(np.ascontiguousarray(c).reshape(-1)))
            clouds.append((flat.view(c.shape), pose))
        m = em.Map(em.Params(**P))
        has_normals = bool(extra.get("flags"))
        m.set_state(h=prior["h"], var=prior["var"], t_last=prior["t_last"].astype(np.float32), t_now=prior["t_now"],
                    **({k: prior[k] for k in ("nx", "ny", "nz")} if has_normals else {}))
        m.update_multi(clouds)
        m.shift(3, -2)
        m.update_multi(clouds)
        got.append((m.state(), m.stats()))
        m.close()
    for s, st in got[1:]:
        for k, v in got[0][0].items():
            assert np.array_equal(v, s[k], equal_nan=True), k
        assert st == got[0][1]


@pytest.mark.parametrize("ray_group", [1, 2, 8, 32])
@pytest.mark.parametrize("order", ["runs", "alternating", "random"])
def test_many_points_in_few_cells(em, ray_group, order):
    """150,000 points of one cell and 60,000 of three others, in runs, in turn and in
    random order among points of other cells: the accumulators' sums, with every
    kind of launch shape, against the float64 means."""
    rng = np.random.default_rng(12)
    W, H = 60, 50
    cells = np.concatenate([np.tile([[17, 20]], (150_000, 1)), np.tile([[18, 20], [0, 0], [59, 49]], (20_000, 1)),
                            np.stack([rng.integers(W, size=30_000), rng.integers(H, size=30_000)], axis=1)])
    if order == "random":
        cells = cells[rng.permutation(len(cells))]
    elif order == "alternating":  # neighbours in a warp in different cells
        cells = cells.reshape(30, -1, 2).transpose(1, 0, 2).reshape(-1, 2)
    xy = (cells + 0.5 + rng.uniform(-0.3, 0.3, cells.shape) - np.array([W, H]) / 2) * R
    p = np.concatenate([xy, rng.uniform(-0.8, -0.3, (len(cells), 1))], axis=1).astype(np.float32)
    maps = [em.Map(em.Params(width=W, height=H, resolution=R, noise_a0=0.005, noise_a2=0.002, ray_step=R)) for _ in range(2)]
    batch = em.Batch(max_maps=2, max_clouds=2, max_points=2 * len(p), max_cells=W * H)
    batch.set_tuning(ray_group=ray_group, fuse_chunk=512, big_thresh=256)
    d = torch.from_numpy(p).cuda()
    batch.update([(m, d, POSE) for m in maps])
    for m in maps:
        m.sync()
        check(m.state(), [(p, cells)], W, H)
        assert m.stats()["points_accepted"] == len(p)
    batch.close()
