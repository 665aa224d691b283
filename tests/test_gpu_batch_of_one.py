"""A batch of one image is set up by the image's own launches, larger ones by the
flat launches of a reload: the same state after the set-up, after a reload and
after iterations, device and host inputs, with the given and the computed
prior."""
import numpy as np
import pytest

from paper_1903_07149_gb300 import build as scalp_build
from paper_1903_07149_gb300 import synth

pytestmark = pytest.mark.gpu

KEYS = ("labels", "n", "sx", "sy", "color", "endpoint")


@pytest.mark.parametrize("H,W,K", [(33, 70, 9), (240, 330, 150)])
@pytest.mark.parametrize("prior", ["input", "gradient"])
@pytest.mark.parametrize("host", [False, True])
def test_set_up_forms(H, W, K, prior, host):
    import torch

    scalp_build.build()
    from paper_1903_07149_gb300 import scalp as S

    rgb, con, _ = synth.small_image(H, W, seed=H, n_cells=12)
    other, con2, _ = synth.small_image(H, W, seed=H + 1, n_cells=5)
    conv = (lambda a: a) if host else (lambda a: torch.from_numpy(a).cuda())
    rgb, con, other, con2 = (conv(a) for a in (rgb, con, other, con2))
    given = prior == "input"
    one = S.Batch([rgb], [con] if given else None, [K], prior=prior)
    two = S.Batch([rgb] * 2, [con] * 2 if given else None, [K] * 2, prior=prior)

    def same():
        a = one.get_state(0)
        for i in range(2):
            b = two.get_state(i)
            for k in KEYS:
                assert np.array_equal(a[k], b[k]), (i, k)

    same()
    one.iterate(3)
    two.iterate(3)
    same()
    one.reload([other], [con2] if given else None)
    two.reload([other] * 2, [con2] * 2 if given else None)
    same()
    one.iterate(2)
    two.iterate(2)
    same()
    a, n = one.labels()
    b, m = two.labels()
    assert n[0] == m[0] == m[1] and np.array_equal(a[0], b[0]) and np.array_equal(a[0], b[1])
    one.close()
    two.close()
