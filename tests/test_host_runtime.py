"""The library's host side without a GPU: its objects linked with a stand-in
for the CUDA runtime (fake_cudart.cpp), driven through the Python binding in a
process of its own.  Kernels are logged, not run; an access past the end of an
allocation ends that process with SIGSEGV."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

PRELUDE = """
import ctypes, sys
import numpy as np
sys.path.insert(0, {root!r})
real = ctypes.CDLL
ctypes.CDLL = lambda path, *a, **k: real({lib!r} if str(path).endswith("libem.so") else path, *a, **k)
from paper_2204_12876_gb300 import em
lib = em.lib
lib.fake_log.restype = ctypes.c_char_p
lib.fake_fail_launch.argtypes = lib.fake_fail_alloc.argtypes = [ctypes.c_long]
em._stream_handle = lambda stream: None

def log(clear=True):
    lines = lib.fake_log().decode().split("\\n")[:-1]
    if clear:
        lib.fake_clear()
    return lines

POSE = np.eye(3, 4, dtype=np.float32)
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """Run a program over the stand-in; its output, and the status it ended with."""
    from paper_2204_12876_gb300 import build
    if not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    lib = str(tmp_path_factory.mktemp("fake") / "libem_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CUDA, "-o", lib,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp"), *objs, "-lpthread"], check=True)
    prelude = PRELUDE.format(root=ROOT, lib=lib)

    def go(program: str):
        p = subprocess.run([sys.executable, "-c", prelude + program], capture_output=True, text=True, timeout=300)
        assert p.returncode == 0, (p.returncode, p.stdout, p.stderr[-2000:])
        return p.stdout
    return go


@pytest.mark.parametrize("sizes", [(1,), (1, 3, 5), (1,) * 63, (0, 7, 2, 0, 9)])
@pytest.mark.parametrize("stride", [3, 4])
def test_host_clouds_stay_inside_the_staging_buffers(run, sizes, stride):
    """The staged clouds start on 16-byte boundaries, so they take more room than
    their floats: calls whose floats just fit (and the calls around them) neither
    write past the pinned buffer nor copy past the device one."""
    run(f"""
sizes, stride = {sizes!r}, {stride}
m = em.Map(em.Params(width=8, height=8))
floats = sum(sizes) * stride
first = 4 * 1024                       # any first call: its slack decides the capacity
m.update_host([(np.zeros((first, 4), np.float32), POSE)])
cap = 4 * first + first + 1024         # floats, with the slack of that call
for short in (0, 1, 2, 3, 4, 8):       # one big cloud before the odd ones makes their total cap - short
    big = (cap - floats - short) // 3
    m.update_host([(np.ones((big, 3), np.float32), POSE)] + [(np.ones((n, stride), np.float32), POSE) for n in sizes])
m.close()
""")


@pytest.mark.parametrize("form", ["update", "uploaded", "batch", "batch_of_one"])
def test_an_update_after_a_failed_launch_starts_with_clear_scratch(run, form):
    """A launch that fails half way leaves sums and marks behind: the next update of
    those maps clears them on its stream before its first kernel, and only that
    one does."""
    run(f"""
form = {form!r}
P = em.Params(width=70, height=50, ray_step=0.04, wall_num_thresh=2, drift_flatness=0.9, flags=em.F_NORMALS)
maps = [em.Map(P), em.Map(P)]
batch = em.Batch(max_maps=2, max_clouds=16, max_points=1000, max_cells=3500, graph=False)
pts = np.zeros((20, 3), np.float32)
clouds = [(pts, POSE)] * (12 if form == "uploaded" else 1)

def update():
    if form.startswith("batch"):
        use = maps if form == "batch" else maps[:1]
        h = (ctypes.c_void_p * len(use))(*[m.handle.value for m in use])
        c = (em._Cloud * len(use))(*[em._cloud_struct(pts, POSE, True) for _ in use])
        em._check(lib.em_update_batch(batch._h, h, c, len(use), None), "em_update_batch")
    else:
        arr = (em._Cloud * len(clouds))(*[em._cloud_struct(p, q, True) for p, q in clouds])
        em._check(lib.em_update_multi(maps[0]._h, arr, len(arr), None), "em_update_multi")

log()
update()
whole = log()
n = sum(l.startswith("launch") for l in whole)
assert n == 5 and not any(l.startswith("memset") for l in whole), whole
cells = 70 * 50
for k in range(2, n + 1):  # the first k - 1 kernels are launched, the k-th is not
    lib.fake_fail_launch(k)
    try:
        update()
        raise SystemExit("the failed launch was not reported")
    except em.EMError as e:
        assert e.code == em.EM_ERR_CUDA
    log()
    update()
    lines = log()
    first = next(i for i, l in enumerate(lines) if l.startswith("launch"))
    sizes = [int(l.split()[2]) for l in lines[:first] if l.startswith("memset")]
    assert not any(l.startswith("memset") for l in lines[first:])
    users = 2 if form == "batch" else 1
    for want in (cells * 32, cells * 4, (cells + 31) // 32 * 4):  # sums; rejected and counted points; marks
        assert sizes.count(want) == users * (2 if want == cells * 4 else 1), (k, sizes)
    update()
    assert log() == whole  # clean again
""")


@pytest.mark.parametrize("wall", [0, 2])
@pytest.mark.parametrize("ray", [0.0, 0.04])
def test_large_maps_hold_memory_for_their_points_not_for_every_cell(run, ray, wall):
    """A map holds, besides its layers, marks and ray thresholds, at most 40 bytes a
    cell for the sums of 512 tiles of 1024 cells (21 MB), and about 80 bytes for
    each point of its largest update, at most 48 a cell: 120 maps of 4096 x 4096
    cells are admitted to 40 GB."""
    run(f"""
for side in (64, 500, 724, 725, 1000, 4096):
    P = em.Params(width=side, height=side, ray_step={ray}, wall_num_thresh={wall})
    m = em.Map(P)
    nc = side * side
    coarse = (side // 8 + 4) ** 2
    layers = nc * (12 + 4 + 1 / 8) + 4 * coarse + 80 * (nc / 1024 + 1) + (1 << 16)
    sums = 40 * min(nc, 1 << 19)
    assert m.info()["device_bytes"] <= layers + sums, (side, m.info())
    for n in (0, 20000, 300000):
        m.reserve(n)
        points = min(80 * 1.25 * n, 48 * nc) if nc > 1 << 19 else 0
        assert m.info()["device_bytes"] <= layers + sums + points, (side, n, m.info())
    m.reserve(5 * nc)  # more points than cells: a sum per cell
    assert m.info()["device_bytes"] <= layers + max(sums, 48 * nc)
    m.close()

srv = em.Server(budget_bytes=40 << 30, max_slots=16, n_streams=1, max_batch_maps=4, max_batch_points=1 << 20,
                max_map_cells=1 << 24, graph=False)
for _ in range(120):
    srv.add_map(em.Params(width=4096, height=4096, ray_step={ray}, wall_num_thresh={wall}))
srv.close()
""")


@pytest.mark.parametrize("maps, clouds, alone", [(1, 1, True), (1, 8, True), (1, 9, False), (2, 1, False)])
def test_autotune_times_the_path_an_update_takes(run, maps, clouds, alone):
    """A batch of one map with the default shape runs as em_update does, with nothing
    to upload; the autotuner times that shape so, and the others as they would run."""
    run(f"""
n_maps, n_clouds, alone, reps = {maps}, {clouds}, {alone}, 3
maps = [em.Map(em.Params(width=40, height=30, ray_step=0.04)) for _ in range(n_maps)]
batch = em.Batch(max_maps=2, max_clouds=16, max_points=1000, max_cells=1200, graph=False)
pts = np.zeros((20, 3), np.float32)
count = n_maps * n_clouds
h = (ctypes.c_void_p * count)(*[maps[i % n_maps].handle.value for i in range(count)])
c = (em._Cloud * count)(*[em._cloud_struct(pts, POSE, True) for _ in range(count)])
uploads = lambda lines: sum(l.startswith("copy 1 ") for l in lines)  # host to device
log()
em._check(lib.em_update_batch(batch._h, h, c, count, None), "em_update_batch")
per_update = uploads(log())
assert per_update == (0 if alone else 2)
t = em._Tuning()
em._check(lib.em_batch_autotune(batch._h, h, c, count, None, reps, ctypes.byref(t)), "em_batch_autotune")
lines = log()
assert sum("k_write" in l for l in lines) == 5 * (reps + 1)  # ray_group 1, 2, 4, 8 and 16
assert uploads(lines) == 2 * (reps + 1) * (4 if alone else 5), uploads(lines)
""")


def test_a_refused_allocation_leaves_no_error_for_the_next_call(run):
    """Every allocation of a map, and of a large map's table, fails in turn: the call
    says so, and the next ones work, those included that ask the runtime for its
    last error after a launch."""
    run("""
large = em.Map(em.Params(width=900, height=900, wall_num_thresh=1))
for k in range(1, 5):
    lib.fake_fail_alloc(k)
    try:
        large.reserve(1000)
        raise SystemExit("a refused allocation was not reported")
    except em.EMError as e:
        assert e.code == em.EM_ERR_OOM
    assert large.info()["point_capacity"] == 0
    em.Map(em.Params(width=20, height=10, ray_step=0.04)).close()
large.reserve(1000)
before = large.info()["device_bytes"]
lib.fake_fail_alloc(2)
try:
    large.reserve(100000)
    raise SystemExit("a refused allocation was not reported")
except em.EMError as e:
    assert e.code == em.EM_ERR_OOM
assert large.info()["point_capacity"] == 0 and large.info()["device_bytes"] < before  # (given back, not half there)
large.update_host([(np.zeros((2000, 3), np.float32), POSE)])
large.close()
k = 0
while True:
    k += 1
    lib.fake_fail_alloc(k)
    try:
        em.Map(em.Params(width=20, height=10, ray_step=0.04, wall_num_thresh=1, flags=em.F_NORMALS)).close()
        break
    except em.EMError as e:
        assert e.code == em.EM_ERR_OOM
    lib.fake_fail_alloc(0)
    em.Map(em.Params(width=20, height=10)).close()
assert k > 10
""")
