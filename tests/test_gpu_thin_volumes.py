"""Supervoxels of thin volumes: the packed form of the assignment's tiles (fewer
than sixteen columns, or one row) and its neighbours, one step from the oracle's
state: labels equal but for near-ties, the sums those of the labels, and the
counted pairs those of the windows."""
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


def pairs_of(st, K, shape):
    """(voxel, cluster) pairs within the windows: |v - s / n|^3 <= N / K on each
    axis, in exact integers."""
    T, H, W = shape
    N, total = T * H * W, 0
    for k in range(len(st["n"])):
        n, places = int(st["n"][k]), 1
        for key, size in (("sx", W), ("sy", H), ("st", T)):
            s = int(st[key][k])
            places *= sum(abs(n * v - s) ** 3 * K <= N * n ** 3 for v in range(size))
        total += places
    return total


@pytest.mark.parametrize("T,H,W,K", [
    (20, 30, 1, 9), (20, 30, 3, 12), (17, 21, 7, 30), (9, 20, 8, 25), (12, 19, 9, 30), (7, 33, 12, 20), (5, 20, 15, 18),
    (40, 1, 50, 20), (33, 1, 8, 9), (1, 1, 400, 12), (1, 400, 1, 12), (400, 1, 1, 12), (1, 30, 5, 6), (2, 9, 13, 5),
    (6, 2, 40, 9), (6, 20, 16, 14), (1, 30, 40, 12), (12, 12, 6, 500), (10, 1, 60, 400)])
def test_step_from_the_oracle(S, T, H, W, K):
    import torch

    rgb, con, _ = synth.small_image(T * H, W, seed=T + H + W, n_cells=max(2, T * H * W // 60))
    rgb, con = rgb.reshape(T, H, W, 3), con.reshape(T, H, W)
    orc = oracle.VSolver(oracle.lab_from_rgb(rgb), con, K)
    orc.assign()
    orc.update()
    st = orc.state()
    seg = S.VoxelSegmenter(torch.from_numpy(rgb).cuda(), torch.from_numpy(con).cuda(), K)
    seg.set_state(dict(labels=st["labels"], n=st["n"], sx=st["sx"], sy=st["sy"], st=st["st"],
                       color=np.stack([st["cL"], st["cA"], st["cB"]], 1),
                       endpoint=np.stack([st["ex"], st["ey"], st["et"]], 1)))
    seg.count_samples(1)
    seg.iterate(1)
    _, pairs = seg.count_samples(0)
    g = seg.get_state()
    seg.close()
    orc.assign()
    lab = orc.labels
    for t, y, x in np.argwhere(g["labels"] != lab):
        Dg, Do = (orc.distance(x, y, t, int(m[t, y, x]))[0] for m in (g["labels"], lab))
        assert abs(Dg - Do) <= 1e-5 * max(Do, 1e-12)
    assert (g["labels"] != lab).sum() <= 0.002 * lab.size + 1
    tt, yy, xx = np.indices(lab.shape)
    flat = g["labels"].ravel()
    n = np.bincount(flat, minlength=len(g["n"]))
    own = n > 0  # (an empty cluster keeps its sums)
    assert np.array_equal(n[own], g["n"][own])
    for key, place in (("sx", xx), ("sy", yy), ("st", tt)):
        assert np.array_equal(np.bincount(flat, place.ravel(), len(n)).astype(np.int64)[own], g[key][own]), key
    assert pairs == pairs_of(st, K, (T, H, W))


# a launch on 147,000 voxels in a plane one column wide against one on as many in
# 49 x 50 x 60: 26 and 20 us; 146 where each tile had a warp for 32 of its places
def test_cost_of_a_column(S):
    import torch

    took = []
    for shape in ((300, 490, 1), (49, 50, 60)):
        gen = torch.Generator(device="cuda").manual_seed(1)
        rgb = torch.randint(0, 240, (*[-(-v // 12) for v in shape], 3), generator=gen, device="cuda", dtype=torch.uint8)
        for axis, v in enumerate(shape):
            rgb = rgb.repeat_interleave(12, axis).narrow(axis, 0, v)
        seg = S.VoxelSegmenter(rgb.contiguous(), None, 100)
        seg.iterate(2)
        seg.profile(1)
        seg.iterate(6)
        ms, launches = seg.profile(0)
        took.append(ms / launches)
        seg.close()
    assert took[0] < 3.0 * took[1], took
