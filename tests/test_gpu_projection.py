"""The projection's search (Eq. 4) over large windows, windows one pixel wide and
clusters whose squared distances leave 64 bits, in both searches that take
whole windows: the endpoint is the pixel of S_k nearest the barycenter, ties to
the smallest index, computed here from the labels and sums in exact integers."""
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


def nearest(place, n, s):
    """Index into `place` (pixels x axes) of the pixel nearest s / n, exactly."""
    d = ((place - np.array(s, np.float64) / n) ** 2).sum(1)
    near = np.flatnonzero(d <= d.min() * (1 + 1e-9) + 1e-9)  # then exactly
    exact = [sum((int(n) * int(x) - int(t)) ** 2 for x, t in zip(place[i], s)) for i in near]
    return int(near[int(np.argmin(exact))])


def check(labels, n, sums, end):
    """Every endpoint is rounded half-up, or projected where its pixel is not of
    S_k; returns the number of projected ones."""
    flat, shape, projected = labels.ravel(), labels.shape, 0
    order = np.argsort(flat, kind="stable")
    bounds = np.searchsorted(flat[order], np.arange(len(n) + 1))
    for k in range(len(n)):
        own = order[bounds[k]:bounds[k + 1]]
        if len(own) == 0:
            continue
        assert len(own) == n[k]
        s = [int(v[k]) for v in sums]  # x, y (, t)
        want = [(2 * v + int(n[k])) // (2 * int(n[k])) for v in s]
        if labels[tuple(want[::-1])] != k:
            place = np.stack(np.unravel_index(own, shape)[::-1], 1)
            want = list(place[nearest(place, n[k], s)])
            projected += 1
        assert list(end[k]) == want, k
    return projected


def stripes(shape):
    """Rows of alternating colours, seven pixels wide, with a little noise: with
    a weak spatial term S_k is a set of stripes and X_k falls on others."""
    import torch

    gen = torch.Generator(device="cuda").manual_seed(shape[-1])
    x = torch.arange(shape[-1], device="cuda") // 7 % 2
    y = torch.arange(shape[-2], device="cuda") // 7 % 2
    on = (x ^ y[:, None]) if min(shape[-2:]) > 1 else x + y[:, None]
    rgb = (on * 180 + 20).to(torch.uint8)[..., None].expand(*shape, 3).clone()
    return rgb + torch.randint(0, 6, rgb.shape, generator=gen, dtype=torch.uint8, device="cuda")


# 64-bit squared distances in windows below and above 2^32 / width pixels, ones
# beyond 64 bits, and one-pixel windows
@pytest.mark.parametrize("H,W,K", [(300, 500, 6), (1700, 1700, 4), (1300, 2700, 2), (30000, 1, 100), (1, 30000, 100)])
@pytest.mark.parametrize("form", ["alone", "batch"])
def test_large_windows(S, H, W, K, form):
    rgb = stripes((H, W))
    if form == "alone":
        a = S.Segmenter(rgb, None, K, m=0.02)
        a.iterate(2)
        g = a.get_state()
    else:
        a = S.Batch([rgb] * 2, None, [K] * 2, m=0.02)
        a.iterate(2)
        g = a.get_state(1)
    a.close()
    assert check(g["labels"], g["n"], (g["sx"], g["sy"]), g["endpoint"]) > 0


@pytest.mark.parametrize("T,H,W,K", [(8, 40, 50, 4), (30, 260, 300, 2), (600, 1, 200, 4), (600, 200, 1, 4)])
def test_large_voxel_windows(S, T, H, W, K):
    a = S.VoxelSegmenter(stripes((T, H, W)), None, K, m=0.02)
    a.iterate(2)
    g = a.get_state()
    a.close()
    assert check(g["labels"], g["n"], (g["sx"], g["sy"], g["st"]), g["endpoint"]) > 0
