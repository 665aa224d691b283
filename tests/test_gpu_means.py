"""Label means (scalp_label_means_static) at the edges of its tiles (64 x 32
pixels, 8 rows per warp) and of its table: ragged sizes, labels to be skipped,
more labels in a tile than the table holds.  Counts and coordinate sums are
exact integers; the colours are within 1e-4 of numpy means of the oracle's FP64
CIELab, as in the other parity tests."""
import numpy as np
import pytest

import oracle
from paper_1903_07149_gb300 import build as scalp_build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["blocks", "pixels", "one"])
@pytest.mark.parametrize("H,W", [(1, 1), (1, 130), (70, 1), (33, 65), (64, 64), (61, 127)])
def test_means_shapes(H, W, kind):
    import torch

    scalp_build.build()
    from paper_1903_07149_gb300 import scalp

    rng = np.random.default_rng(H * 1000 + W)
    rgb = rng.integers(0, 256, (H, W, 3), dtype=np.uint8)
    if kind == "pixels":  # a label of its own for every pixel
        lab = rng.permutation(H * W).reshape(H, W)
    elif kind == "one":
        lab = np.zeros((H, W), int)
    else:  # blocks with noise; labels outside [0, n) are skipped
        lab = np.kron(rng.integers(-1, 9, (H // 6 + 1, W // 10 + 1)), np.ones((6, 10), int))[:H, :W]
        lab = np.where(rng.random((H, W)) < 0.05, rng.integers(-2, 12, (H, W)), lab)
    n = min(H * W, 65536) if kind == "pixels" else 8
    out = torch.full((n, 6), -1.0, dtype=torch.float64, device="cuda")
    d_rgb, d_lab = torch.from_numpy(rgb).cuda(), torch.from_numpy(lab.astype(np.int32)).cuda()
    scalp.scalp_label_means_static(d_rgb.data_ptr(), 0, d_lab.data_ptr(), H, W, n, out.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
    got = out.cpu().numpy()
    keep = (lab >= 0) & (lab < n)
    k = lab[keep]
    cnt = np.bincount(k, minlength=n)
    assert np.array_equal(got[:, 0], cnt)
    some = cnt > 0
    ys, xs = np.nonzero(keep)
    assert np.array_equal(got[some, 4], np.bincount(k, xs, n)[some] / cnt[some])
    assert np.array_equal(got[some, 5], np.bincount(k, ys, n)[some] / cnt[some])
    for i, plane in enumerate(oracle.lab_from_rgb(rgb)):
        ref = np.bincount(k, np.asarray(plane).reshape(H, W)[keep], n)[some] / cnt[some]
        assert np.all(np.abs(got[some, 1 + i] - ref) <= 1e-4 * np.maximum(np.abs(ref), 1))
    assert np.all(got[~some] == 0.0)
