"""Point queries: counts that are no multiple of the points per thread, bases
that allow no vector access, points in and out of order, on voxel faces,
outside every block and not finite; and resets that leave nothing behind."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _map(voxel, layer=0, storage=0, seed=0, max_blocks=1 << 12):
    import paper_2311_00626_gb300 as gt
    rng = np.random.default_rng(seed)
    keys = np.unique(rng.integers(-6, 6, (300, 3)), axis=0).astype(np.int32)
    D = rng.uniform(-3 * voxel, 3 * voxel, (len(keys), 512)).astype(np.float32)
    W = rng.integers(0, 50, (len(keys), 512)).astype(np.float32)
    m = gt.TsdfMap(voxel, 4, 100.0, storage=storage, layer=layer, max_blocks=max_blocks)
    m.import_blocks(keys, D, W)
    return m, m.export()


def _points(voxel, rng, n):
    p = rng.uniform(-60 * voxel, 60 * voxel, (n, 3)).astype(np.float32)
    grid = (rng.integers(-50, 50, (n, 3)).astype(np.float32) * np.float32(voxel)).astype(np.float32)
    pick = np.arange(n) % 5
    p[pick == 1] = grid[pick == 1]                        # on voxel faces
    p[pick == 2] = np.nextafter(grid, -np.inf)[pick == 2]
    p[(pick == 3) & (rng.random(n) < 0.3)] = 0.0
    run = (np.arange(n) // 13) % 2 == 0                   # runs along x, as a grid is queried
    p[run, 1:] = p[run][:1, 1:] if run.any() else 0.0
    odd = np.float32([np.nan, np.inf, -np.inf, 1e38, -1e38, 1e-45, -1e-45, -0.0, 1e7, -1e-30])
    where = rng.random((n, 3)) < 0.02
    p[where] = odd[rng.integers(0, len(odd), where.sum())]
    return p


def _expect(points, voxel, exported, fill):
    keys, *vals = exported
    at = {tuple(k): i for i, k in enumerate(keys)}
    with np.errstate(all="ignore"):
        g = np.floor(points / np.float32(voxel))
    out = [np.full((len(points),) + v.shape[2:], fill, v.dtype) for v in vals]
    for i, q in enumerate(g):
        if not (np.abs(q) < 8.0 * (1 << 20)).all():
            continue
        c = q.astype(np.int64)
        b = at.get(tuple(int(x) for x in c >> 3))
        if b is not None:
            l = int((c[0] & 7) + 8 * (c[1] & 7) + 64 * (c[2] & 7))
            for o, v in zip(out, vals):
                o[i] = v[b, l]
    return out


@pytest.mark.parametrize("n", [1, 3, 4, 5, 127, 512, 515, 2001])
@pytest.mark.parametrize("voxel,storage,layer", [(0.05, 0, 0), (0.02, 1, 0), (0.1, 2, 0), (0.3, 0, 1), (1e-30, 0, 0)])
def test_query_matches_export(n, voxel, storage, layer):
    import torch
    m, exported = _map(voxel, layer, storage)
    p = _points(voxel, np.random.default_rng(n), n)
    want = _expect(p, voxel, exported, 0.0)
    for shift in (0, 1):  # with and without 16-byte bases
        pts = torch.cat([torch.zeros(shift), torch.from_numpy(p).flatten()]).cuda()[shift:].view(n, 3)
        dist, weight = (torch.full((n + shift,), 7.0, device="cuda")[shift:] for _ in range(2))
        m.query(pts, dist, weight)
        np.testing.assert_array_equal(dist.cpu().numpy(), want[0])
        np.testing.assert_array_equal(weight.cpu().numpy(), want[1])
    m.close()


@pytest.mark.parametrize("n", [1, 6, 1029])
def test_color_and_esdf_queries_match_exports(n):
    import torch
    import paper_2311_00626_gb300 as gt
    import synth
    w = synth.config_tiny()
    f = w.frames[0]
    d = torch.from_numpy(f.depth).cuda()
    c = torch.randint(0, 1 << 24, f.depth.shape, dtype=torch.int32, device="cuda")
    m = gt.TsdfMap(w.voxel_size, 4, 100.0, layer=gt.LAYER_COLOR, max_blocks=1 << 12)
    m.integrate_color(f.sensor, f.T, d, c)
    keys, rgb, W = m.export_color()
    rng = np.random.default_rng(n)
    p = ((keys[rng.integers(0, len(keys), n)] + rng.uniform(-0.1, 1.1, (n, 3))) * 8 * w.voxel_size).astype(np.float32)
    want = _expect(p, w.voxel_size, (keys, rgb, W), 0.0)
    for shift in (0, 1):
        pts = torch.cat([torch.zeros(shift), torch.from_numpy(p).flatten()]).cuda()[shift:].view(n, 3)
        out = torch.full((3 * n + shift,), 7.0, device="cuda")[shift:].view(n, 3)
        wt = torch.full((n + shift,), 7.0, device="cuda")[shift:]
        m.query_color(pts, out, wt)
        np.testing.assert_array_equal(out.cpu().numpy(), want[0])
        np.testing.assert_array_equal(wt.cpu().numpy(), want[1])
    m.close()
    m = gt.TsdfMap(w.voxel_size, 4, 100.0, max_blocks=1 << 12)
    m.integrate(f.sensor, f.T, d)
    m.esdf_update()
    keys, st = m.esdf_export()
    off = [((st >> (9 * a)) & 511).astype(np.int64) for a in range(3)]
    off = [np.where(o >= 256, o - 512, o) for o in off]
    r = np.sqrt(np.float32(off[0] ** 2 + off[1] ** 2 + off[2] ** 2))
    r = np.where(st & (1 << 29), r, np.float32(64)).astype(np.float32)
    v = np.where(st & (1 << 30), -r, r) * np.float32(w.voxel_size)
    v = np.where(st & (1 << 27), v, np.nan).astype(np.float32)
    want = _expect(p, w.voxel_size, (keys, v), np.nan)
    for shift in (0, 1):
        pts = torch.cat([torch.zeros(shift), torch.from_numpy(p).flatten()]).cuda()[shift:].view(n, 3)
        out = torch.full((n + shift,), 7.0, device="cuda")[shift:]
        m.esdf_query(pts, out)
        np.testing.assert_array_equal(out.cpu().numpy(), want[0])
    m.close()


@pytest.mark.parametrize("max_blocks", [1, 7, 33, 1 << 12])
def test_reset_leaves_nothing_behind(max_blocks):
    """After a reset a map (its table, pool, changed flags, ESDF states) behaves like a new one."""
    import paper_2311_00626_gb300 as gt
    rng = np.random.default_rng(max_blocks)
    n = min(max_blocks, 60)
    keys = np.stack([np.arange(n), np.zeros(n), np.zeros(n)], 1).astype(np.int32)
    D = rng.uniform(-0.2, 0.2, (2, n, 512)).astype(np.float32)
    W = np.ones((n, 512), np.float32)
    a = gt.TsdfMap(0.05, 4, 100.0, max_blocks=max_blocks)
    a.import_blocks(keys, D[0], W)
    a.esdf_update()
    a.reset()
    assert a.num_blocks() == 0 and a.esdf_stats() == dict(iterations=0, swept=0, pulled=0, cleared=0)
    b = gt.TsdfMap(0.05, 4, 100.0, max_blocks=max_blocks)
    half = max(1, n // 2)
    for m in (a, b):
        m.import_blocks(keys[:half], D[1, :half], W[:half])
        m.esdf_update()
        assert m.sync() == 0
    for x, y in zip(a.export() + a.esdf_export(), b.export() + b.esdf_export()):
        np.testing.assert_array_equal(x, y)
    assert a.esdf_stats() == b.esdf_stats()
    a.close()
    b.close()
