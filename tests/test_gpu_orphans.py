"""Projections (Eq. 4) when some pixels lie in no window and keep their label:
S_k then reaches outside cluster k's window, and the nearest pixel of S_k may
be such a pixel.  Windows, sums and projections are exact integers, so the
endpoints equal the oracle's wherever the pixel sets agree, and batched and
persistent launches equal each image solved alone bit for bit."""
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


def stranded_state(shape, K, x_k, seed):
    """An oracle solver of a (H, W) image or (T, H, W) volume whose barycenters
    all lie near column x_k, so that the columns more than r to the right are in
    no window, with labels in narrow vertical bands: every cluster keeps pixels
    there and its next barycenter falls between bands."""
    rng = np.random.default_rng(seed)
    if len(shape) == 2:
        rgb, con, _ = synth.small_image(*shape, seed=seed)
        orc = oracle.Solver(oracle.lab_from_rgb(rgb), con, K)
    else:
        rgb, con, _ = synth.voronoi_video(*shape, 6, seed=seed)
        orc = oracle.VSolver(oracle.lab_from_rgb(rgb), con, K)
    st = orc.state()
    W, Ke = shape[-1], orc.Keff
    band = (np.arange(W) // 3) % Ke
    st["labels"] = np.ascontiguousarray(np.broadcast_to(band, shape)).astype(np.int32)
    for key in ("sy", "st")[:len(shape) - 1]:
        st[key][:] = st[key] * 100 // st["n"]
    st["n"][:] = 100
    st["sx"][:] = 100 * x_k + rng.integers(-99, 100, Ke)
    st["ex"][:] = x_k
    orc.set_state(st)
    return rgb, con, orc, orc.state()


# a few hundred orphans, and more than one pass of a CTA over their list
@pytest.mark.parametrize("H,W,K,x_k", [(6, 100, 3, 15), (60, 200, 3, 15), (60, 430, 6, 15)])
def test_endpoints_with_orphans(S, H, W, K, x_k):
    import torch

    rgb, con, orc, st = stranded_state((H, W), K, x_k, seed=W)
    seg = S.Segmenter(torch.from_numpy(rgb).cuda(), torch.from_numpy(con).cuda(), orc.K)
    seg.set_state(dict(labels=st["labels"], n=st["n"], sx=st["sx"], sy=st["sy"],
                       color=np.stack([st["cL"], st["cA"], st["cB"]], 1),
                       endpoint=np.stack([st["ex"], st["ey"]], 1)))
    orc.assign()
    assert orc.orphans > 0
    lab = orc.labels.copy()
    orc.update()
    assert orc.projections > 0  # (of this update)
    seg.iterate(1)
    g = seg.get_state()
    differ = g["labels"] != lab
    assert differ.mean() <= 0.001
    same = np.setdiff1d(np.arange(orc.Keff), np.unique(np.concatenate([g["labels"][differ], lab[differ]])))
    assert len(same) > 0
    assert np.array_equal(g["endpoint"][same], orc.endpoints()[same])
    seg.close()


def test_voxel_endpoints_with_orphans(S):
    import torch

    rgb, con, orc, st = stranded_state((4, 24, 90), 8, 12, seed=7)
    seg = S.VoxelSegmenter(torch.from_numpy(rgb).cuda(), torch.from_numpy(con).cuda(), orc.K)
    seg.set_state(dict(labels=st["labels"], n=st["n"], sx=st["sx"], sy=st["sy"], st=st["st"],
                       color=np.stack([st["cL"], st["cA"], st["cB"]], 1),
                       endpoint=np.stack([st["ex"], st["ey"], st["et"]], 1)))
    orc.assign()
    assert orc.orphans > 0
    lab = orc.labels.copy()
    orc.update()
    assert orc.projections > 0  # (of this update)
    seg.iterate(1)
    g = seg.get_state()
    differ = g["labels"] != lab
    assert differ.mean() <= 0.001
    same = np.setdiff1d(np.arange(orc.Keff), np.unique(np.concatenate([g["labels"][differ], lab[differ]])))
    assert len(same) > 0
    s2 = orc.state()
    ref = np.stack([s2["ex"], s2["ey"], s2["et"]], 1)
    assert np.array_equal(g["endpoint"][same], ref[same])
    seg.close()


# flat cells and a weak spatial term (m = 1): clusters drift and strand pixels;
# (H, W, K, cells, gradient, seed)
DRIFT = [(101, 79, 153, 36, False, 33), (72, 123, 300, 30, True, 314)]


def drift_image(i):
    H, W, _, n, gradient, seed = DRIFT[i]
    rgb, con, _ = synth.small_image(H, W, seed=seed, n_cells=n, gradient=gradient)
    return rgb, con


@pytest.mark.parametrize("mode", ["flat", "persistent"])
@pytest.mark.parametrize("copies", [4, 40])
def test_batches_with_orphans_equal_alone(S, mode, copies):
    """Few images (CTAs per image) and 80 (the work lists: more than four
    queued clusters per CTA, so warps search)."""
    import torch

    for i, (H, W, K, _, _, _) in enumerate(DRIFT):
        rgb, con = drift_image(i)
        orc = oracle.Solver(oracle.lab_from_rgb(rgb), con, K, m=1.0)
        seen = 0
        for _ in range(5):
            orc.assign()
            seen += orc.orphans
            orc.update()
        assert seen > 0
    made = [drift_image(i) for i in range(len(DRIFT))] * copies
    rgbs = [torch.from_numpy(m[0]).cuda() for m in made]
    cons = [torch.from_numpy(m[1]).cuda() for m in made]
    Ks = [d[2] for d in DRIFT] * copies
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        alone = []
        for i in range(len(DRIFT)):
            s = S.Segmenter(rgbs[i], cons[i], Ks[i], m=1.0, stream=stream)
            s.iterate(6)
            alone.append(s.get_state())
            s.close()
        b = S.Batch(rgbs, cons, Ks, m=1.0, stream=stream)
        b.set_launch(mode)
        b.iterate(6)
        for i in range(len(rgbs)):
            g = b.get_state(i)
            for k in ("labels", "n", "sx", "sy", "color", "endpoint"):
                assert np.array_equal(g[k], alone[i % len(DRIFT)][k]), (i, k)
        b.close()
