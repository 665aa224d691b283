"""The cluster update on eight lanes a cluster (up to 24,576 clusters a launch) and
on one thread: a single image on either side of the line against the same image
in a batch of three, which lies above it, bit for bit."""
import numpy as np
import pytest

from paper_1903_07149_gb300 import build as scalp_build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,K", [(384, 1024, 24576), (384, 1040, 24960), (300, 700, 9000), (512, 1024, 32768)])
def test_forms_agree(H, W, K):
    import torch

    scalp_build.build()
    from paper_1903_07149_gb300 import scalp as S

    gen = torch.Generator(device="cuda").manual_seed(H)
    rgb = torch.randint(0, 256, (H // 9 + 1, W // 11 + 1, 3), generator=gen, dtype=torch.uint8, device="cuda")
    rgb = rgb.repeat_interleave(9, 0).repeat_interleave(11, 1)[:H, :W].contiguous()
    a = S.Segmenter(rgb, None, K)
    keff = a.info.Keff
    assert (keff <= 24576) == (K <= 24576)
    assert 3 * keff > 24576
    a.iterate(3)
    g = a.get_state()
    a.close()
    b = S.Batch([rgb] * 3, None, [K] * 3)
    b.iterate(3)
    for i in range(3):
        h = b.get_state(i)
        for k in ("labels", "n", "sx", "sy", "color", "endpoint"):
            assert np.array_equal(g[k], h[k]), (i, k)
    b.close()
