"""LiDAR projection of voxel pairs against the one-by-one IEEE form: the same
scan with every length scaled by a power of two, so that the coordinates leave
the range of the pair forms.  Each FP32 operation scales exactly, so blocks and
weights are the same and distances scale exactly."""
from __future__ import annotations

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2311_00626_gb300 as gt  # noqa: E402


def _scan(power, T, ranges, **opts):
    """The scan in units of 2^-power voxels' worth: everything times 2^power."""
    k = 2.0 ** power
    s = {"kind": "lidar", "n_az": ranges.shape[1], "n_el": ranges.shape[0], "theta_start": -math.pi,
         "phi_start": math.radians(50.0), "el_fov": math.radians(80.0), "min_range": 0.5 * k, "max_range": 40.0 * k}
    m = gt.TsdfMap(0.25 * k, max_blocks=1 << 15, **opts)
    T = T.copy()
    T[:3, 3] *= k
    d = torch.from_numpy(ranges * np.float32(k)).cuda()
    m.integrate(s, T, d)
    gt.integrate_batch([m.handle], [gt.frame_desc(0, s, T, d)] * 2)
    assert m.sync() == 0
    keys, D, W = m.export()
    m.close()
    return keys, D, W


@pytest.mark.parametrize("opts", [{}, {"lidar_nearest": True}, {"weighting": gt.WEIGHT_DROPOFF},
                                  {"layer": gt.LAYER_OCCUPANCY}])
@pytest.mark.parametrize("pose", ["centre", "corner", "turned"])
def test_pairs_equal_the_one_by_one_form(pose, opts):
    rng = np.random.default_rng(11)
    n_el, n_az = 33, 257
    j, i = np.mgrid[0:n_el, 0:n_az]
    r = (6.0 + 3.0 * np.sin(i * 2 * math.pi / n_az * 3) + 0.1 * j + 0.02 * rng.normal(size=(n_el, n_az)))
    r[rng.random(r.shape) < 0.05] = 0.0
    r[:, 100:120] = 25.0
    T = np.eye(4)
    if pose == "centre":  # sensor on a voxel centre: coordinates that are exactly 0, the sensor's own voxel
        T[:3, 3] = 0.125
        r[:, 30:40] = 0.6
    elif pose == "turned":
        a, b = 0.7, -0.3
        T[:3, :3] = (np.array([[math.cos(a), -math.sin(a), 0], [math.sin(a), math.cos(a), 0], [0, 0, 1]])
                     @ np.array([[1, 0, 0], [0, math.cos(b), -math.sin(b)], [0, math.sin(b), math.cos(b)]]))
        T[:3, 3] = rng.uniform(-5, 5, 3)
    r = r.astype(np.float32)
    keys, D, W = _scan(0, T, r, **opts)
    assert len(keys) > 200 and ((W > 0).sum() > 20000 or "layer" in opts)
    scale_d = "layer" not in opts
    for power in (28, -36):  # coordinates beyond 2^30; all below 2^-30
        k2, D2, W2 = _scan(power, T, r, **opts)
        np.testing.assert_array_equal(k2, keys)
        np.testing.assert_array_equal(W2, W)
        np.testing.assert_array_equal(D2, D * np.float32(2.0 ** power) if scale_d else D)


@pytest.mark.parametrize("n_az,n_el,fov", [(1024, 64, 45.0), (257, 2, 20.0), (2048, 128, 120.0), (1, 33, 90.0)])
def test_pair_cells_equal_the_one_by_one_cells(n_az, n_el, fov):
    """Weighted maps find a voxel's beam cell one voxel at a time.  With the
    drop-off weights a voxel in front of it has weight 1, so after one scan it
    holds the same distance as in a constant-weight map, whose cells come from
    voxel pairs, if the sample positions are the same."""
    rng = np.random.default_rng(n_az)
    j, i = np.mgrid[0:n_el, 0:n_az]
    r = 6.0 + 2.0 * np.sin(i * 2 * math.pi / n_az * 3) + 0.05 * j + 0.02 * rng.normal(size=i.shape)
    r[rng.random(r.shape) < 0.02] = 0.0
    s = {"kind": "lidar", "n_az": n_az, "n_el": n_el, "theta_start": -math.pi,
         "phi_start": math.radians(90.0 - fov / 2), "el_fov": math.radians(fov), "min_range": 0.5, "max_range": 30.0}
    T = np.eye(4)
    T[:2, :2] = [[math.cos(0.3), -math.sin(0.3)], [math.sin(0.3), math.cos(0.3)]]
    T[:3, 3] = [0.31, -0.2, 0.77]
    d = torch.from_numpy(r.astype(np.float32)).cuda()
    out = []
    for weighting in (gt.WEIGHT_CONSTANT, gt.WEIGHT_DROPOFF):
        m = gt.TsdfMap(0.1, weighting=weighting)
        m.integrate(s, T, d)
        assert m.sync() == 0
        out.append(m.export())
        m.close()
    (k, D, W), (k2, D2, W2) = out
    np.testing.assert_array_equal(k, k2)
    one = W2 == 1
    assert one.sum() > 50 and (W[one] == 1).all()
    np.testing.assert_array_equal(D[one], D2[one])
