"""The first call of the ESDF layer or the mesher with too little device memory
left: it returns TSDF_ERR_CUDA, nothing later uses what was not allocated, and
the same call succeeds once there is memory."""
from __future__ import annotations

import contextlib
import ctypes

import numpy as np
import pytest

from tests.esdf_inputs import V, tsdf_region

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2311_00626_gb300 as gt  # noqa: E402

ERR_CUDA = -2
EPS = float(V)
BLOCKS = 1 << 24  # 64 MB for a list of block indices


@contextlib.contextmanager
def _little_memory():
    """Less than 56 MB of free device memory."""
    hold = []
    for size in (4 << 30, 256 << 20, 32 << 20):
        while torch.cuda.mem_get_info()[0] > size + (24 << 20):
            hold.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
    assert torch.cuda.mem_get_info()[0] < 56 << 20
    try:
        yield
    finally:
        hold.clear()
        torch.cuda.empty_cache()


def _map():
    keys, D, W, _ = tsdf_region((0, 0, 0), (3, 3, 4), lambda c: c[..., 2] - 0.43)
    g = gt.TsdfMap(EPS, max_blocks=BLOCKS, storage=gt.STORAGE_FP16)
    g.import_blocks(keys, D, W)
    return g, (keys, D, W)


def test_esdf_without_memory():
    g, blocks = _map()
    pts = torch.from_numpy(((blocks[0] * 8 + 4.5) * EPS).astype(np.float32)).cuda()
    dist = torch.empty(len(pts), device="cuda")
    with _little_memory():
        for _ in range(2):
            with pytest.raises(gt.TsdfError) as e:
                g.esdf_update(EPS, 1e-4, 60)
            assert e.value.code == ERR_CUDA
        for call in (lambda: g.esdf_query(pts, dist), g.esdf_export):  # there is no layer
            with pytest.raises(gt.TsdfError):
                call()
        g.reset()
        assert g.sync() == 0
    g.import_blocks(*blocks)
    g.esdf_update(EPS, 1e-4, 60)
    small = gt.TsdfMap(EPS, max_blocks=1 << 10, storage=gt.STORAGE_FP16)
    small.import_blocks(*blocks)
    small.esdf_update(EPS, 1e-4, 60)
    for a, b in zip(g.esdf_export(), small.esdf_export()):
        np.testing.assert_array_equal(a, b)
    g.close()
    small.close()


def test_mesh_without_memory():
    g, blocks = _map()
    n = ctypes.c_int64()
    pos = torch.empty((1 << 14, 9), device="cuda")

    def mesh():
        return gt.lib().map_mesh(g.handle, 1e-4, 0, pos.data_ptr(), None, None, len(pos), ctypes.byref(n), None)

    with _little_memory():
        assert mesh() == ERR_CUDA
        assert mesh() == ERR_CUDA
    assert mesh() == 0
    assert n.value > 1000
    g.close()
