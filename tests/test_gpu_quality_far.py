"""Boundary recall with radii above fifteen pixels: the disk's search against
plain numpy, and its cost beside the masks' (radii up to fifteen)."""
import time

import numpy as np
import pytest

from paper_1903_07149_gb300 import build as scalp_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch

    assert torch.cuda.is_available()
    scalp_build.build()
    from paper_1903_07149_gb300 import scalp

    scalp.load()
    return scalp


def maps(H, W, a, b):
    """Superpixels of a x a cells, segments of b x b cells shifted by a third."""
    y, x = np.mgrid[:H, :W]
    lab = (y // a) * (W // a + 1) + x // a
    gt = ((y + b // 3) // b) * (W // b + 2) + (x + b // 3) // b
    return lab.astype(np.int32), gt.astype(np.int32)


def boundary(m):
    e = np.zeros(m.shape, bool)
    d = m[:, 1:] != m[:, :-1]
    e[:, 1:] |= d
    e[:, :-1] |= d
    d = m[1:] != m[:-1]
    e[1:] |= d
    e[:-1] |= d
    return e


# radii with pixels exactly at eps (17: 8, 15; 25: 7, 24; 20: 12, 16), beyond the
# image, and infinite
@pytest.mark.parametrize("H,W,a,b", [(90, 130, 41, 53), (1, 300, 70, 90), (300, 1, 70, 90), (40, 300, 300, 17),
                                     (257, 61, 45, 300)])
@pytest.mark.parametrize("eps", [15.0, 15.5, 16.0, 17.0, 20.0, 25.0, 25.000001, 40.3, 100.0, 1e6, 1e300, float("inf")])
def test_recall(S, H, W, a, b, eps):
    import torch

    lab, gt = maps(H, W, a, b)
    sy, sx = np.nonzero(boundary(lab))
    gy, gx = np.nonzero(boundary(gt))
    hit = 0
    for y, x in zip(gy, gx):
        hit += len(sy) > 0 and bool(np.any(np.sqrt(((sy - y) ** 2 + (sx - x) ** 2).astype(np.float64)) < eps))
    want = hit / len(gy) if len(gy) else 1.0
    got = S.quality_metrics(torch.from_numpy(lab).cuda(), torch.from_numpy(gt).cuda(), eps=eps)
    assert got["br"] == want


# 321 x 481, six superpixels: at eps = 40 1.4 ms against 0.09 at eps = 15 (16
# times); 83 ms (970 times) where the warps took their rows one after the other
def test_cost_of_far_radii(S):
    import torch

    lab, gt = (torch.from_numpy(m).cuda() for m in maps(321, 481, 170, 61))
    took = []
    for eps in (15.0, 40.0):
        best = 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            S.quality_metrics(lab, gt, eps=eps)
            best = min(best, time.perf_counter() - t0)
        took.append(best)
    assert took[1] < 120 * took[0], took
