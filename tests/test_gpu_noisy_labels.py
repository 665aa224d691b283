"""Connectivity enforcement of labels that are noise: long chains of small
components, against the oracle, and their cost beside that of coherent labels."""
import time

import numpy as np
import pytest

import oracle
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


PATTERNS = {
    "random": lambda rng, y, x, k: rng.integers(0, k, y.shape),
    "two": lambda rng, y, x, k: rng.integers(0, 2, y.shape) % k,
    "rows": lambda rng, y, x, k: y % k,
    "columns": lambda rng, y, x, k: x % k,
    "checker": lambda rng, y, x, k: (x + y) % k,
    "blocks": lambda rng, y, x, k: (y // 5 * 7919 + x // 5 * 31) % k,
    "one": lambda rng, y, x, k: 0 * x,
}


def with_labels(S, H, W, K, pattern, stream=None):
    import torch

    seg = S.Segmenter(torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda"), None, K, stream=stream)
    st = seg.get_state()
    y, x = np.mgrid[:H, :W]
    st["labels"] = PATTERNS[pattern](np.random.default_rng(H + W), y, x, len(st["n"])).astype(np.int32)
    seg.set_state(st)
    return seg, st["labels"]


@pytest.mark.parametrize("H,W,K", [(40, 50, 9), (1, 9000, 5), (9000, 1, 5), (700, 2, 3), (129, 64, 60), (200, 333, 3),
                                   (211, 127, 2000)])
@pytest.mark.parametrize("pattern", sorted(PATTERNS))
def test_chains(S, H, W, K, pattern):
    seg, lab = with_labels(S, H, W, K, pattern)
    out, n = seg.labels(enforce=True)
    ref, nref = oracle.connectivity(lab, K)
    seg.close()
    assert n == nref and np.array_equal(out, ref)


# 1080 x 1920, a random label per pixel against blocks of 5 x 5: 2.5 ms against
# 0.18 (14 times); 16.9 against 0.34 (50 times) with two loads a hop in turn
def test_cost_of_noise(S):
    import torch

    took = []
    for pattern in ("random", "blocks"):
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            seg, _ = with_labels(S, 1080, 1920, 2000, pattern, stream)
            out = torch.empty((1080, 1920), dtype=torch.int32, device="cuda")
            best = 1e9
            for _ in range(6):
                stream.synchronize()
                t0 = time.perf_counter()
                seg.labels(enforce=True, out=out)
                best = min(best, time.perf_counter() - t0)
            seg.close()
        took.append(best)
    assert took[0] < 26 * took[1], took
