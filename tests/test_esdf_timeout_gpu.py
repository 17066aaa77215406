"""An ESDF update whose grid-wide wait runs out (made to by the wait-test
hook: the wait is bounded and returns, nothing hangs), and the recovery that
map_reset promises."""
from __future__ import annotations

import numpy as np
import pytest

from tests.esdf_inputs import V, tsdf_region

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import paper_2311_00626_gb300 as gt  # noqa: E402

TIMEOUT = -4
EPS = float(V)
RANGE = 120  # voxels


def _wall():
    """A wall at one end of a row of 12 x 2 x 2 blocks: the distances cross
    the row block by block, one exchange each."""
    return tsdf_region((0, 0, 0), (12, 2, 2), lambda c: c[..., 0] - 0.21)[:3]


def _gave_up(g, blocks):
    """Import the blocks, then an update that is made to give up."""
    g.import_blocks(*blocks)
    gt.map_wait_test(g.handle, 1)
    with pytest.raises(gt.TsdfError) as e:
        g.esdf_update(EPS, 1e-4, RANGE)
    assert e.value.code == TIMEOUT
    gt.map_wait_test(g.handle, 0)


def test_reset_restores_the_layer_after_an_update_gave_up():
    blocks = _wall()
    g = gt.TsdfMap(EPS, max_blocks=1 << 12)
    o = oracle.EsdfOracle(EPS, EPS, 1e-4, RANGE)
    o.update(*blocks, np.ones(len(blocks[0]), bool))
    want = o.export()
    assert o.counters()["iterations"] >= 8
    for _ in range(2):
        _gave_up(g, blocks)
        assert g.sync() == TIMEOUT
        g.reset()
        g.import_blocks(*blocks)
        g.esdf_update(EPS, 1e-4, RANGE)
        assert g.sync() == 0
        for a, b in zip(g.esdf_export(), want):
            np.testing.assert_array_equal(a, b)
        assert g.esdf_stats() == o.counters()
        g.reset()
    g.close()
    o.close()


def test_a_half_done_layer_is_not_read_out():
    """Between the update that gave up and the reset, the states are a mix of
    two buffers and of iterations: reading them is refused."""
    blocks = _wall()
    g = gt.TsdfMap(EPS, max_blocks=1 << 12)
    g.import_blocks(*blocks)
    g.esdf_update(EPS, 1e-4, RANGE)
    pts = torch.from_numpy(((blocks[0] * 8 + 4.5) * EPS).astype(np.float32)).cuda()
    dist = torch.empty(len(pts), device="cuda")
    g.reset()
    _gave_up(g, blocks)
    for call in (lambda: g.esdf_query(pts, dist), g.esdf_export, lambda: g.esdf_update(EPS, 1e-4, RANGE)):
        with pytest.raises(gt.TsdfError) as e:
            call()
        assert e.value.code == TIMEOUT
    g.reset()
    assert len(g.esdf_export()[0]) == 0
    g.esdf_query(pts, dist)
    assert torch.isnan(dist).all()
    g.close()
