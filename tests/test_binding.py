"""The Python binding's marshalling, without a GPU."""
import ctypes
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")


class DeviceCloud:
    """What the binding asks of a CUDA tensor."""
    is_cuda, dtype = True, torch.float32

    def __init__(self, n, stride, ptr):
        self.shape, self._ptr = (n, stride), ptr

    def is_contiguous(self):
        return True

    def dim(self):
        return 2

    def data_ptr(self):
        return self._ptr


@pytest.mark.parametrize("map_id", [3, True, np.int64(3), np.uint8(3), 3.0, np.float32(3), "3", -1, (1 << 32) + 3])
def test_requests_take_any_map_id_that_is_an_int(monkeypatch, map_id):
    """Map ids are taken by int(), as they always were: numpy's and whole floats too."""
    from paper_2204_12876_gb300 import build
    build.build()
    from paper_2204_12876_gb300 import em
    seen = []

    def submit(handle, reqs, n, ready, tickets):
        for i in range(n):
            r = reqs[i]
            seen.append((r.map_id, r.n_clouds, r.clouds_on_host, r.read_mask, r.clouds[0].points, r.clouds[0].n,
                         r.clouds[0].stride, list(r.clouds[r.n_clouds - 1].pose)))
            tickets[i] = 10 + i
        return 0

    monkeypatch.setattr(em, "lib", types.SimpleNamespace(em_server_submit_many=submit))
    s = object.__new__(em.Server)
    s._h, s._keep = None, {}
    poses = [np.arange(12.0), np.arange(12, dtype=np.float32).reshape(3, 4) + 1, list(range(2, 14))]
    clouds = [(DeviceCloud(5 + k, 3 + k % 2, 4096 * (k + 1)), q) for k, q in enumerate(poses)]
    assert s.submit_many([(map_id, clouds, None), (0, clouds[1:], None)]) == [10, 11]
    want = ctypes.c_int32(int(map_id)).value
    assert seen == [(want, 3, 0, 0, 4096, 5, 3, [float(v) for v in range(2, 14)]),
                    (0, 2, 0, 0, 8192, 6, 4, [float(v) for v in range(2, 14)])]
