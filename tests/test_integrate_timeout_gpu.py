"""An integration launch whose bounded wait for a work-list entry runs out
(made to by the wait-test hook; it returns after some 0.1 s): every map of
the call reports it, and map_reset recovers."""
from __future__ import annotations

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2311_00626_gb300 as gt  # noqa: E402

TIMEOUT = -4


@pytest.mark.parametrize("n_maps,n_frames", [(1, 1), (3, 6), (1, 40)])
def test_every_map_of_the_call_reports_the_wait(n_maps, n_frames):
    frames = synth.config_room(n_frames=300).frames[:n_frames]
    dev = [torch.from_numpy(np.ascontiguousarray(f.depth)).cuda() for f in frames]
    maps = [gt.TsdfMap(0.05, max_blocks=1 << 14) for _ in range(n_maps)]

    def call():
        if n_frames == 1:
            maps[0].integrate(frames[0].sensor, frames[0].T, dev[0])
        else:
            gt.integrate_batch([m.handle for m in maps], [gt.frame_desc(i % n_maps, f.sensor, f.T, d)
                                                          for i, (f, d) in enumerate(zip(frames, dev))])
        torch.cuda.synchronize()

    call()
    assert all(m.sync() == 0 for m in maps)
    want = [m.export() for m in maps]
    for m in maps:
        m.reset()
    gt.map_wait_test(maps[0].handle, 1)
    call()
    assert [m.sync() for m in maps] == [TIMEOUT] * n_maps
    gt.map_wait_test(maps[0].handle, 0)
    for m in maps:
        m.reset()
    call()
    assert all(m.sync() == 0 for m in maps)
    for m, w in zip(maps, want):
        for a, b in zip(m.export(), w):
            np.testing.assert_array_equal(a, b)
        m.close()
