"""The ESDF update on a stream that has a part of the GPU's SMs (a green
context): its cooperative launch takes as many CTAs as fit there."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

from tests.esdf_inputs import V, tsdf_region

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import paper_2311_00626_gb300 as gt  # noqa: E402

EPS = float(V)


class _Partition:
    """A stream of a green context with about `sms` SMs (CUDA driver API)."""

    def __init__(self, sms):
        d = self.driver = ctypes.CDLL("libcuda.so.1")
        torch.zeros(1, device="cuda")  # the primary context is active
        # CUdevResource: int type, 92 bytes, then the SM count first in a 48-byte union
        res, part, rest = ((ctypes.c_uint32 * 36)() for _ in range(3))
        n, desc, self.ctx, self.stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
        for err in (d.cuDeviceGetDevResource(0, res, 1),
                    d.cuDevSmResourceSplitByCount(part, ctypes.byref(n), res, rest, 0, sms),
                    d.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1),
                    d.cuGreenCtxCreate(ctypes.byref(self.ctx), desc, 0, 1),
                    d.cuGreenCtxStreamCreate(ctypes.byref(self.stream), self.ctx, 1, 0)):
            if err:
                pytest.skip(f"no green contexts here (driver error {err})")
        self.sms = part[24]

    def close(self):
        self.driver.cuStreamDestroy_v2(self.stream)
        self.driver.cuGreenCtxDestroy(self.ctx)


@pytest.mark.parametrize("sms", [8, 32])
def test_update_on_a_part_of_the_gpu(sms):
    keys, D, W, _ = tsdf_region((-3, -2, -4), (5, 4, 2),
                                lambda c: np.linalg.norm(c - np.array([-0.31, 0.2, -0.6]), axis=-1) - 0.4)
    o = oracle.EsdfOracle(EPS, EPS, 1e-4, 60)
    o.update(keys, D, W, np.ones(len(keys), bool))
    p = _Partition(sms)
    assert p.sms < torch.cuda.get_device_properties(0).multi_processor_count
    g = gt.TsdfMap(EPS, max_blocks=1 << 12)
    g.import_blocks(keys, D, W)
    gt.map_esdf_update(g.handle, EPS, 1e-4, 60, stream=p.stream.value)
    torch.cuda.synchronize()
    for a, b in zip(g.esdf_export(), o.export()):
        np.testing.assert_array_equal(a, b)
    assert g.esdf_stats() == o.counters()
    g.close()
    o.close()
    p.close()
