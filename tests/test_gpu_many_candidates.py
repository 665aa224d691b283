"""Tiles with more candidates than shared memory holds (grid steps of about two
and three pixels): the per-pixel path of single images, batches in both launch
modes and both storages, bit for bit, and near-ties only against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1903_07149_gb300 import build as scalp_build
from paper_1903_07149_gb300 import synth

pytestmark = pytest.mark.gpu

KEYS = ("labels", "n", "sx", "sy", "color", "endpoint")


@pytest.mark.parametrize("H,W,r", [(70, 101, 2.0), (70, 101, 2.6), (97, 64, 3.0), (33, 400, 1.5)])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_per_pixel_path(H, W, r, storage):
    import torch

    scalp_build.build()
    from paper_1903_07149_gb300 import scalp as S

    K = int(H * W / r / r)
    rgb, con, _ = synth.small_image(H, W, seed=H + W, n_cells=40)
    d_rgb, d_con = torch.from_numpy(rgb).cuda(), torch.from_numpy(con).cuda()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        a = S.Segmenter(d_rgb, d_con, K, storage=storage, stream=stream)
        a.iterate(3)
        g = a.get_state()
        a.close()
        for mode in ("flat", "persistent"):
            b = S.Batch([d_rgb] * 3, [d_con] * 3, [K] * 3, storage=storage, stream=stream)
            b.set_launch(mode)
            b.iterate(3)
            for i in range(3):
                h = b.get_state(i)
                for k in KEYS:
                    assert np.array_equal(g[k], h[k]), (mode, i, k)
            b.close()
    if storage == "f32":  # one step from the oracle's state
        orc = oracle.Solver(oracle.lab_from_rgb(rgb), con, K)
        orc.iterate(1)
        st = orc.state()
        with torch.cuda.stream(stream):
            a = S.Segmenter(d_rgb, d_con, K, stream=stream)
            a.set_state(dict(labels=st["labels"], n=st["n"], sx=st["sx"], sy=st["sy"],
                             color=np.stack([st["cL"], st["cA"], st["cB"]], 1),
                             endpoint=np.stack([st["ex"], st["ey"]], 1)))
            a.iterate(1)
            g = a.get_state()
            a.close()
        orc.assign()
        for y, x in np.argwhere(g["labels"] != orc.labels):
            Dg, Do = (orc.distance(x, y, int(m[y, x]))[0] for m in (g["labels"], orc.labels))
            assert (Dg - Do) / max(Do, 1e-12) < 1e-5
        assert (g["labels"] != orc.labels).mean() <= 0.001
