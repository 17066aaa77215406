"""The running average D <- D + (s - D) / (W + 1) in FP32: one rounding after the
product with the reciprocal, for every sensor and launch form."""
from __future__ import annotations

import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2311_00626_gb300 as gt  # noqa: E402


def _frames(kind):
    rng = np.random.default_rng(5)
    if kind == "pinhole":
        w, h = 160, 120
        s = {"kind": "pinhole", "fu": 140.0, "fv": 140.0, "cu": 79.5, "cv": 59.5, "width": w, "height": h}
        j, i = np.mgrid[0:h, 0:w]
        surface = 1.5 + 0.2 * np.sin(i / 31.0) + 0.1 * np.cos(j / 17.0)
    else:
        w, h = 512, 32
        s = {"kind": "lidar", "n_az": w, "n_el": h, "theta_start": -math.pi, "phi_start": math.radians(67.5),
             "el_fov": math.radians(45.0), "min_range": 0.5, "max_range": 30.0}
        j, i = np.mgrid[0:h, 0:w]
        surface = 2.0 + 0.2 * np.sin(i * 2 * math.pi / w)
    return s, [torch.from_numpy((surface + e * (1 + 0.01 * rng.random((h, w)))).astype(np.float32)).cuda()
               for e in (0.0, 0.021, -0.013)]


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("kind", ["pinhole", "lidar"])
def test_the_average_is_rounded_once(kind, batch):
    s, (a, b, c) = _frames(kind)

    def fused(*images):
        m = gt.TsdfMap(0.05)
        if batch:
            gt.integrate_batch([m.handle], [gt.frame_desc(0, s, np.eye(4), d) for d in images])
        else:
            for d in images:
                m.integrate(s, np.eye(4), d)
        assert m.sync() == 0
        keys, D, W = m.export()
        m.close()
        return {tuple(k): (x, w) for k, x, w in zip(keys, D, W)}

    two, one, three = fused(a, b), fused(c), fused(a, b, c)
    keys = [k for k in three if k in two and k in one]
    D2, W2 = (np.stack([two[k][i] for k in keys]) for i in (0, 1))
    s3, W1 = (np.stack([one[k][i] for k in keys]) for i in (0, 1))  # D = s with W = 1: 1 / 1 is exact
    D3, W3 = (np.stack([three[k][i] for k in keys]) for i in (0, 1))
    ok = (W2 == 2) & (W1 == 1) & (W3 == 3)
    assert ok.sum() > 10000
    D2, s3, D3 = D2[ok], s3[ok], D3[ok]
    third = np.float32(1) / np.float32(3)  # the reciprocal is within one unit of it
    cand = [np.nextafter(third, np.float32(0)), third, np.nextafter(third, np.float32(1))]
    # D + e r in FP64 is exact but for its last bits (24 + 24 bits beside D's 24)
    once = [(D2.astype(np.float64) + (s3 - D2).astype(np.float64) * np.float64(r)).astype(np.float32) for r in cand]
    twice = [D2 + (s3 - D2) * r for r in cand]
    assert any(np.array_equal(D3, x) for x in once)
    assert not any(np.array_equal(D3, x) for x in twice)  # the inputs tell the two apart
