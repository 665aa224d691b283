"""Batches around the number of images up to which the projection's work lists
fit a launch's shared memory (3,007; batches of 3,036 to 3,071 once did not
launch), in both launch modes: every image as in a batch of four."""
import numpy as np
import pytest

from paper_1903_07149_gb300 import build as scalp_build
from paper_1903_07149_gb300 import synth

pytestmark = pytest.mark.gpu

KEYS = ("labels", "n", "sx", "sy", "color", "endpoint")
SHAPES = [(9, 14, 5), (16, 16, 4), (5, 33, 6), (20, 11, 9)]


@pytest.fixture(scope="module")
def S():
    import torch

    assert torch.cuda.is_available()
    scalp_build.build()
    from paper_1903_07149_gb300 import scalp

    scalp.load()
    return scalp


def solve(S, count, mode):
    import torch

    made = [synth.small_image(H, W, seed=H, n_cells=4)[:2] for H, W, _ in SHAPES]
    dev = [(torch.from_numpy(r).cuda(), torch.from_numpy(c).cuda()) for r, c in made]
    pick = [i % len(SHAPES) for i in range(count)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        b = S.Batch([dev[i][0] for i in pick], [dev[i][1] for i in pick], [SHAPES[i][2] for i in pick], stream=stream)
        b.set_launch(mode)
        b.iterate(3)
        at = sorted(set(range(min(count, 4))) | {count // 2, count - 2, count - 1})
        states = {i: b.get_state(i) for i in at}
        b.close()
    return states


@pytest.mark.parametrize("mode", ["flat", "persistent"])
@pytest.mark.parametrize("count", [3007, 3008, 3035, 3036, 3039, 3040, 3071, 3072])
def test_work_lists_limit(S, count, mode):
    few = solve(S, 4, "flat")
    for i, g in solve(S, count, mode).items():
        for k in KEYS:
            assert np.array_equal(g[k], few[i % 4][k]), (i, k)
