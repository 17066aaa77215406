"""The allocation kernel for pinhole tiles by pixel patches against the row
kernel: walking every pixel (what walk statistics select) must give the same
blocks and, through them, the same voxels, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (3, 5), (4, 4), (31, 33), (64, 64), (63, 65), (65, 31), (333, 7), (130, 66), (256, 192)]


def _pose(rng, far):
    q = rng.normal(size=4)
    a, b, c, d = q / np.linalg.norm(q)
    T = np.eye(4)
    T[:3, :3] = [[a * a + b * b - c * c - d * d, 2 * (b * c - a * d), 2 * (b * d + a * c)],
                 [2 * (b * c + a * d), a * a - b * b + c * c - d * d, 2 * (c * d - a * b)],
                 [2 * (b * d - a * c), 2 * (c * d + a * b), a * a - b * b - c * c + d * d]]
    T[:3, 3] = rng.uniform(-far, far, 3)
    return T


def _depth(rng, kind, w, h):
    j, i = np.mgrid[0:h, 0:w]
    wall = 2.0 + 0.8 * np.sin(i / 37.0) + 0.5 * np.cos(j / 23.0)
    if kind == "smooth":  # a curved surface with a little noise and missing pixels
        d = wall + 0.01 * rng.normal(size=(h, w))
        d[rng.random((h, w)) < 0.05] = 0.0
    elif kind == "edges":  # steps between a near and a far surface
        d = np.where(((i // 9) + (j // 7)) % 3 == 0, 0.6, wall * 2)
        d[(i + j) % 11 == 0] = 0.0
    elif kind == "noise":  # every pixel at another depth: most patches fail the test
        d = rng.uniform(0.01, 20.0, (h, w))
    else:  # missing, negative, non-finite and extreme values between valid ones
        d = np.where(rng.random((h, w)) < 0.5, wall, 0.0)
        bad = np.array([np.nan, np.inf, -np.inf, -1.0, 1e-38, 1e-45, 3.4028235e38, 1e6, 0.0])
        pick = rng.random((h, w)) < 0.2
        d[pick] = bad[rng.integers(0, len(bad), pick.sum())]
    return d.astype(np.float32)


def _run(frames, voxel, tile_h, walk_all, batch):
    import torch
    import paper_2311_00626_gb300 as gt
    m = gt.TsdfMap(voxel, 4, 100.0, max_blocks=1 << 19, alloc_tile_h=tile_h)
    gt.map_walk_stats(m.handle, walk_all)
    if batch:
        gt.integrate_batch([m.handle], [gt.frame_desc(0, s, T, d) for s, T, d in frames])
    else:
        for s, T, d in frames:
            m.integrate(s, T, d)
    torch.cuda.synchronize()
    assert m.sync() == 0
    out = m.export(), m.stats()["block_frame_pairs"], m.stats()["voxel_updates"]
    m.close()
    return out


@pytest.mark.parametrize("tile_h", [16, 32])
@pytest.mark.parametrize("voxel,far", [(0.05, 3.0), (0.02, 300.0), (0.004, 1.0), (0.5, 20.0)])
@pytest.mark.parametrize("kind", ["smooth", "edges", "noise", "invalid"])
def test_patches_meet_the_blocks_of_every_pixel(kind, voxel, far, tile_h):
    import torch
    rng = np.random.default_rng([ord(kind[0]), int(voxel * 1000), tile_h])
    for batch in (False, True):
        frames = []
        for n, (w, h) in enumerate(SIZES):
            f = 0.8 * max(w, h)
            s = {"kind": "pinhole", "fu": -f if n % 4 == 3 else f, "fv": f * 1.1, "cu": (w - 1) / 2 + 0.3,
                 "cv": (h - 1) / 2, "width": w, "height": h}
            d = torch.from_numpy(_depth(rng, kind, w, h)).cuda()
            if n % 3 == 2:  # a base that is not 16-byte aligned: no vector loads
                d = torch.cat([torch.zeros(1, device="cuda"), d.flatten()])[1:].view(h, w)
            frames.append((s, _pose(rng, far), d))
        got, pairs, upd = _run(frames, voxel, tile_h, False, batch)
        want, wpairs, wupd = _run(frames, voxel, tile_h, True, batch)
        assert pairs == wpairs and upd == wupd
        for a, b in zip(got, want):
            np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))


def test_patches_beside_lidar_frames():
    """A batch of cameras and LiDARs: camera tiles by patches, LiDAR tiles by rows."""
    import math
    import torch
    rng = np.random.default_rng(3)
    frames = []
    for w, h in SIZES[4:]:
        s = {"kind": "pinhole", "fu": 0.8 * w, "fv": 0.8 * w, "cu": (w - 1) / 2, "cv": (h - 1) / 2, "width": w,
             "height": h}
        frames.append((s, _pose(rng, 2.0), torch.from_numpy(_depth(rng, "smooth", w, h)).cuda()))
        li = {"kind": "lidar", "n_az": 101 + w, "n_el": 5 + h % 13, "theta_start": -math.pi,
              "phi_start": math.radians(67.5), "el_fov": math.radians(45.0), "min_range": 0.5, "max_range": 30.0}
        r = rng.uniform(0.0, 32.0, (li["n_el"], li["n_az"])).astype(np.float32)
        frames.append((li, _pose(rng, 2.0), torch.from_numpy(r).cuda()))
    for tile_h in (16, 32):
        got, pairs, upd = _run(frames, 0.05, tile_h, False, True)
        want, wpairs, wupd = _run(frames, 0.05, tile_h, True, True)
        assert pairs == wpairs and upd == wupd
        for a, b in zip(got, want):
            np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
