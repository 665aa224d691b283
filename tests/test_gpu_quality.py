"""Quality metrics (Eq. 5-8) on the GPU against the oracle, on oracle-made
decompositions of synthetic images whose Voronoi cells are the ground truth."""
import numpy as np
import pytest

import oracle
from paper_1903_07149_gb300 import build as scalp_build
from paper_1903_07149_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch

    assert torch.cuda.is_available()
    scalp_build.build()
    from paper_1903_07149_gb300 import scalp

    scalp.load()
    return scalp


@pytest.mark.parametrize("seed,K", [(51, 60), (52, 250)])
def test_quality_matches_oracle(S, seed, K):
    import torch

    rgb, C, cells = synth.small_image(180, 260, seed=seed, n_cells=10)
    s, out, n = oracle.solve(rgb, C, K, iters=4)
    ref = oracle.quality(out, cells)
    got = S.quality_metrics(torch.from_numpy(out).cuda(), torch.from_numpy(cells).cuda())
    assert got["br"] == ref["br"] and got["asa"] == ref["asa"] and got["ue"] == ref["ue"]
    assert got["co"] == pytest.approx(ref["co"], rel=1e-12)


def test_quality_of_gpu_decomposition_is_sane(S):
    import torch

    rgb, C, cells = synth.small_image(240, 320, seed=53, n_cells=12)
    seg = S.Segmenter(torch.from_numpy(rgb).cuda(), torch.from_numpy(C).cuda(), 300)
    seg.iterate(10)
    out = torch.empty((240, 320), dtype=torch.int32, device="cuda")
    seg.labels(enforce=True, out=out)
    q = S.quality_metrics(out, torch.from_numpy(cells).cuda())
    assert 0.9 < q["asa"] <= 1.0 and 0.0 <= q["ue"] < 0.5 and 0.5 < q["br"] <= 1.0
    assert 0.2 < q["co"] < np.pi / 4 + 1e-9
    seg.close()


def _reference(lab, gt, eps):
    """The metrics by plain numpy, any eps."""
    h, w = lab.shape

    def edges(m):
        return [np.pad(m[:, 1:] != m[:, :-1], ((0, 0), (1, 0))), np.pad(m[:, 1:] != m[:, :-1], ((0, 0), (0, 1))),
                np.pad(m[1:] != m[:-1], ((1, 0), (0, 0))), np.pad(m[1:] != m[:-1], ((0, 1), (0, 0)))]

    ys, xs = np.nonzero(np.any(edges(lab), 0))
    gy, gx = np.nonzero(np.any(edges(gt), 0))
    if len(gy):
        d2 = np.full(len(gy), np.inf)
        for y, x in zip(ys, xs):
            d2 = np.minimum(d2, (gy - y) ** 2.0 + (gx - x) ** 2.0)
        br = np.count_nonzero(np.sqrt(d2) < eps) / len(gy)
    else:
        br = 1.0
    n, m = lab.max() + 1, gt.max() + 1
    ov = np.bincount((lab * m + gt).ravel(), minlength=n * m).reshape(n, m)
    area = ov.sum(1)
    rim = np.zeros((h, w), int)
    rim[0] += 1; rim[-1] += 1; rim[:, 0] += 1; rim[:, -1] += 1
    rim += np.sum(edges(lab), 0)
    perim = np.bincount(lab.ravel(), rim.ravel(), n)
    ue = np.where(ov > 0, area[:, None] - ov, 0).sum()
    a = area[area > 0].astype(float)
    co = (4 * np.pi * a * a / perim[area > 0] ** 2).sum()
    return {"br": br, "asa": ov.max(1).sum() / (h * w), "ue": ue / (h * w), "co": co / (h * w)}


# ragged strips (32 columns x 16 rows), one row, one column, one pixel; disks of
# every kind: the pixel alone, half-widths up to the mask's 15, and beyond it
@pytest.mark.parametrize("H,W", [(1, 1), (1, 70), (50, 1), (33, 65), (16, 32), (47, 97)])
@pytest.mark.parametrize("eps", [0.5, 1.0, 2.0, 4.3, 15.0, 15.5])
def test_quality_shapes_and_radii(S, H, W, eps):
    import torch

    rng = np.random.default_rng(H * 1000 + W)
    blk = rng.integers(0, 12, (H // 7 + 1, W // 9 + 1))
    lab = np.kron(blk, np.ones((7, 9), int))[:H, :W]
    lab = np.where(rng.random((H, W)) < 0.03, rng.integers(0, 12, (H, W)), lab).astype(np.int32)
    gt = np.kron(rng.integers(0, 3, (H // 29 + 1, W // 41 + 1)), np.ones((29, 41), int))[:H, :W].astype(np.int32)
    got = S.quality_metrics(torch.from_numpy(lab).cuda(), torch.from_numpy(gt).cuda(), eps=eps)
    # the same maps 4 bytes off a 16-byte boundary (the counts' vector loads)
    a, b = (torch.from_numpy(np.concatenate([[m.max() + 5], m.ravel()]).astype(np.int32)).cuda()[1:].view(H, W)
            for m in (lab, gt))
    assert S.quality_metrics(a, b, eps=eps) == got
    ref = _reference(lab, gt, eps)
    assert got["br"] == ref["br"] and got["asa"] == ref["asa"] and got["ue"] == ref["ue"], (got, ref)
    assert got["co"] == pytest.approx(ref["co"], rel=1e-12)
