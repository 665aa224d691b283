"""The prior's normalisation over outputs without gaps (one row of all pixels,
whatever the width) and with rows at every alignment: the same bits, nothing
outside the rows."""
import numpy as np
import pytest

from paper_1903_07149_gb300 import build as scalp_build

pytestmark = pytest.mark.gpu


# around the 2,048 pixels of a CTA, one row and one column, larger odd widths
@pytest.mark.parametrize("H,W", [(1, 2047), (1, 2049), (2049, 1), (683, 3), (205, 10), (45, 91), (321, 481), (1079, 1919)])
def test_rows_and_gaps(H, W):
    import torch

    scalp_build.build()
    from paper_1903_07149_gb300 import scalp as S

    gen = torch.Generator(device="cuda").manual_seed(H + W)
    rgb = torch.randint(0, 256, (H, W, 3), generator=gen, dtype=torch.uint8, device="cuda")
    want = None
    for offset, pad in ((0, (-W) % 4), (0, 0), (0, 1), (1, 0), (2, 1), (3, (-W - 3) % 4)):
        stride = offset + W + pad
        flat = torch.full((H * stride + 8,), -1.0, device="cuda")
        base = flat[:H * stride].view(H, stride)
        S.gradient_prior(rgb, out=base[:, offset:offset + W])
        got = base[:, offset:offset + W].cpu().numpy()
        if want is None:
            want = got
            assert got.max() == 1.0
        assert np.array_equal(got, want), (offset, pad)
        base[:, offset:offset + W] = -1.0
        assert bool((flat == -1.0).all())
    # a dense output that starts off a 16-byte boundary
    flat = torch.full((H * W + 8,), -1.0, device="cuda")
    S.gradient_prior(rgb, out=flat[1:1 + H * W].view(H, W))
    assert np.array_equal(flat[1:1 + H * W].view(H, W).cpu().numpy(), want)
    assert float(flat[0]) == -1.0 and bool((flat[1 + H * W:] == -1.0).all())


# up to 2,560 tiles of 32 x 32 take a maximum each where the workspace has the
# room (2,550, 2,560 and 2,600 here): the bits of the one cleared word
@pytest.mark.parametrize("H,W", [(1600, 1632), (1280, 2048), (1280, 2049)])
def test_maximum_per_tile(H, W):
    import ctypes

    import torch

    scalp_build.build()
    from paper_1903_07149_gb300 import scalp as S

    gen = torch.Generator(device="cuda").manual_seed(W)
    rgb = torch.randint(0, 256, (H, W, 3), generator=gen, dtype=torch.uint8, device="cuda")
    a = S.gradient_prior(rgb)
    L = S.load()
    nbytes = L.scalp_gradient_prior_workspace_bytes(H, W, 1, 1)
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    b = torch.empty((H, W), device="cuda")
    img = S.scalp_image(H, W, rgb.data_ptr(), 0, 1)
    rc = L.scalp_gradient_prior(ctypes.byref(img), b.data_ptr(), W, 1, torch.cuda.current_stream().cuda_stream,
                                ws.data_ptr(), nbytes)
    assert rc == S.SCALP_OK and torch.equal(a, b) and float(a.max()) == 1.0
