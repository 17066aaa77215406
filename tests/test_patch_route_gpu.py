"""Which batches are allocated by pixel patches, seen from the names of the
kernels that ran, and cases where the patch test's geometry degenerates or most
cells lie outside a tile's window: block sets and voxels equal to walking every
pixel, bit for bit."""
from __future__ import annotations

import math

import numpy as np
import pytest

from tests.test_patch_alloc_gpu import _run

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _kernels(f):
    """Names of the CUDA kernels that f() launches, and its result.  (A process's
    first trace may come back empty.)"""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            out = f()
            torch.cuda.synchronize()
        names = " ".join(e.name for e in p.events())
        if names:
            return names, out
    pytest.skip("no kernel trace here")


def _camera(w, h, f=None, cu=None, cv=None):
    f = f or 0.8 * max(w, h)
    return {"kind": "pinhole", "fu": f, "fv": f, "cu": (w - 1) / 2 if cu is None else cu,
            "cv": (h - 1) / 2 if cv is None else cv, "width": w, "height": h}


def _turned(axis, quarter):
    T = np.eye(4)
    c, s = [1, 0, -1, 0][quarter], [0, 1, 0, -1][quarter]
    a, b = [(1, 2), (0, 2), (0, 1)][axis]
    T[a, a], T[a, b], T[b, a], T[b, b] = c, -s, s, c
    return T


def _compare(frames, voxel, tile_h, batch=True):
    names, got = _kernels(lambda: _run(frames, voxel, tile_h, False, batch))
    assert "patch_alloc_kernel" in names
    names, want = _kernels(lambda: _run(frames, voxel, tile_h, True, batch))
    assert "patch_alloc_kernel" not in names
    assert got[1:] == want[1:]
    for a, b in zip(got[0], want[0]):
        np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))


@pytest.mark.parametrize("axis,quarter", [(0, 0), (0, 1), (0, 3), (1, 1), (1, 2), (2, 1)])
@pytest.mark.parametrize("off", [0.0, 0.05 * 8 * 3])
def test_rays_along_the_axes(axis, quarter, off):
    """Axis-aligned poses, principal point at a patch's centre: the patch's
    central direction is 0 on two axes.  off: sensor on a block corner."""
    T = _turned(axis, quarter)
    T[:3, 3] = off
    frames = []
    for cu, cv in ((33.5, 65.5), (64.0, 64.0), (65.5, 33.5)):
        j, i = np.mgrid[0:130, 0:130]
        d = (1.0 + 0.3 * np.sin(i / 9.0) * np.cos(j / 7.0)).astype(np.float32)
        for depth in (d, np.full_like(d, 1.2)):
            frames.append((_camera(130, 130, 100.0, cu, cv), T, torch.from_numpy(depth).cuda()))
    _compare(frames, 0.05, 32)


@pytest.mark.parametrize("voxel", [0.05, 0.02, 0.01, 0.004])
def test_surfaces_on_both_sides_of_the_window(voxel):
    """Alternating near and far pixels: up to all cells outside the 32-block
    window, hundreds to thousands of them per tile."""
    rng = np.random.default_rng(int(voxel * 1000))
    frames = []
    for k, (w, h) in enumerate([(64, 64), (130, 70), (256, 192)]):
        j, i = np.mgrid[0:h, 0:w]
        near = ((i // 5 + j // 3) % 2 == 0) if k else ((i + j) % 2 == 0)
        d = np.where(near, 0.5 + 0.002 * i, 9.0 - 0.01 * j) + 0.01 * rng.normal(size=(h, w))
        T = np.eye(4)
        T[:3, 3] = rng.uniform(-2, 2, 3)
        frames.append((_camera(w, h), T, torch.from_numpy(d.astype(np.float32)).cuda()))
    _compare(frames, voxel, 32)


@pytest.mark.parametrize("w,h,f,voxel,n,patches", [
    (1600, 1000, 1280.0, 0.05, 1, True),     # above the 3 << 19 pixels of the rule
    (640, 480, 525.0, 0.05, 4, False),       # below
    (640, 480, 525.0, 0.01, 8, True),        # a voxel spans 5.25 pixels at 1 m
    (640, 480, 470.0, 0.01, 8, False),       # 4.7
    (1600, 1000, 1280.0, 0.009, 1, False),   # finer than 1 cm: 11.5 of 15
    (1600, 1000, -1280.0, 0.009, 7, True),   # 11.5 of 7.5 in a launch of 11 M pixels
    (1600, 1000, 1700.0, 0.009, 1, True),    # 15.3
])
def test_which_launches_take_patches(w, h, f, voxel, n, patches):
    j, i = np.mgrid[0:h, 0:w]
    d = torch.from_numpy((1.0 + 0.2 * np.sin(i / 90.0) + 0.1 * np.cos(j / 70.0)).astype(np.float32)).cuda()
    T = np.eye(4)
    frames = []
    for k in range(n):
        T[0, 3] = 0.01 * k
        frames.append((_camera(w, h, f), T.copy(), d))
    names, got = _kernels(lambda: _run(frames, voxel, 0, False, n > 1))
    assert ("patch_alloc_kernel" in names) == patches
    want = _run(frames, voxel, 0, True, n > 1)
    assert got[1:] == want[1:]
    for a, b in zip(got[0], want[0]):
        np.testing.assert_array_equal(a.view(np.int32), b.view(np.int32))
