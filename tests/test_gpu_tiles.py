"""The forms of the assignment's tiles, of the cluster update and of the grid:
each single image against the same image as a batch of one (32 x 32 tiles of
512 threads whatever the size), bit for bit."""
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


def step(H, W, r):
    return max(1, int(round(H * W / (r * r))))


# 16 x 16 tiles (at most 192 tiles of 32 x 32, r <= 24): exact, one over and one
# under tile multiples, one row or column, few and many CTAs per SM, candidates
# up to the per-pixel path; 1024 threads (at most 152 tiles, r > 24); 512 threads
# just above both limits
@pytest.mark.parametrize("H,W,K", [
    (16, 16, 4), (15, 17, 6), (32, 48, 12), (33, 49, 12), (1, 200, 9), (130, 1, 7), (16, 16, 200), (40, 40, 800),
    (96, 160, 60), (200, 300, step(200, 300, 8)), (250, 330, step(250, 330, 23.9)), (384, 512, step(384, 512, 20)),
    (96, 160, step(96, 160, 30)), (250, 330, step(250, 330, 60)), (33, 33, 1),
    (384, 513, step(384, 513, 20)), (384, 512, step(384, 512, 24.5))])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_tile_forms_agree(S, H, W, K, storage):
    import torch

    rgb, con, _ = synth.small_image(H, W, seed=H * 7 + W, n_cells=max(2, H * W // 1500))
    d_rgb, d_con = torch.from_numpy(rgb).cuda(), torch.from_numpy(con).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        seg = S.Segmenter(d_rgb, d_con, K, storage=storage, stream=stream)
        seg.iterate(4)
        a = seg.get_state()
        out, n = seg.labels(enforce=True)
        b = S.Batch([d_rgb], [d_con], [K], storage=storage, stream=stream)
        b.iterate(4)
        g = b.get_state(0)
        outs, ns = b.labels(enforce=True)
        for k in ("labels", "n", "sx", "sy", "color", "endpoint"):
            assert np.array_equal(a[k], g[k]), k
        assert n == ns[0] and np.array_equal(out, outs[0])
        seg.close()
        b.close()


def test_many_clusters_one_step(S):
    """More clusters than the update gives eight lanes each: counts, sums and
    endpoints equal the oracle's for clusters whose pixel sets agree."""
    import torch

    H, W, K = 500, 700, 36000
    rgb, con, _ = synth.small_image(H, W, seed=99, n_cells=60)
    orc = oracle.Solver(oracle.lab_from_rgb(rgb), con, K)
    assert orc.Keff > 32768
    seg = S.Segmenter(torch.from_numpy(rgb).cuda(), torch.from_numpy(con).cuda(), K)
    seg.iterate(1)
    g = seg.get_state()
    orc.assign()
    lab = orc.labels.copy()
    orc.update()
    differ = g["labels"] != lab
    assert differ.mean() <= 0.001
    same = np.setdiff1d(np.arange(orc.Keff), np.unique(np.concatenate([g["labels"][differ], lab[differ]])))
    for k in ("n", "sx", "sy"):
        assert np.array_equal(g[k][same], getattr(orc, k)[same]), k
    assert np.array_equal(g["endpoint"][same], orc.endpoints()[same])
    seg.close()


def test_more_tile_rows_than_a_grid_has(S):
    """65,537 rows of tiles (the grid turns flat): a column of pixels gives the
    labels of the same pixels as a row (the same windows, samples and order)."""
    import torch

    n = 32 * 65536 + 5
    rng = np.random.default_rng(3)
    rgb = np.repeat(rng.integers(0, 256, (n // 50 + 1, 3), dtype=np.uint8), 50, axis=0)[:n]
    con = rng.random(n).astype(np.float32) * 0.2
    K = 40000
    states = []
    for shape in ((n, 1), (1, n)):
        seg = S.Segmenter(torch.from_numpy(rgb.reshape(*shape, 3)).cuda(), torch.from_numpy(con.reshape(shape)).cuda(), K)
        seg.iterate(3)
        states.append((seg.get_state(), seg.labels(enforce=True)[1]))
        seg.close()
    (a, na), (b, nb) = states
    assert np.array_equal(a["labels"].ravel(), b["labels"].ravel()) and na == nb
    assert np.array_equal(a["n"], b["n"]) and np.array_equal(a["sy"], b["sx"]) and np.array_equal(a["color"], b["color"])
