"""The kernels' forms beyond their size and alignment limits: connectivity with
more chunks than its numbering sums itself, volumes with more tiles than the
one-launch lists scan, prior outputs that 16-byte accesses cannot serve."""
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


# 8,192 chunks of 4,096 pixels are numbered without a scan kernel, 8,193 with it
@pytest.mark.parametrize("H,W", [(8192, 4096), (8193, 4096)])
def test_connectivity_chunk_limit(S, H, W):
    import torch

    K = 3000
    seg = S.Segmenter(torch.zeros((H, W, 3), dtype=torch.uint8, device="cuda"), None, K)
    st = seg.get_state()
    rng = np.random.default_rng(H)
    base = rng.integers(0, seg.info.Keff, size=(H // 61 + 1, W // 61 + 1), dtype=np.int32)
    lab = np.repeat(np.repeat(base, 61, axis=0), 61, axis=1)[:H, :W].copy()
    noise = rng.integers(0, H * W, size=H * W // 50)
    lab.ravel()[noise] = rng.integers(0, seg.info.Keff, size=noise.size, dtype=np.int32)
    st["labels"] = lab
    seg.set_state(st)
    out, n = seg.labels(enforce=True)
    ref, nref = oracle.connectivity(lab, K)
    assert n == nref and np.array_equal(out, ref)
    seg.close()


# 12,032 tiles of 16 x 8 x 4 voxels are listed beside the projection, 12,033 in
# launches of their own (12,287 once did not launch).  A line of voxels along t
# has the paths, candidates and sums of the same line along x, which takes a
# quarter of the tiles, so the two agree bit for bit.  (An FP64 comparison says
# less here: at 48,000 an FP32 barycenter is good to 0.002, which moves D by
# more than the 1e-5 that near-ties are allowed elsewhere.)
@pytest.mark.parametrize("n", [4 * 12032, 4 * 12032 + 1, 4 * 12287])
def test_voxel_list_limit(S, n):
    import torch

    rgb, con, _ = synth.small_image(n, 1, seed=5, n_cells=2000)
    out = []
    for shape in ((n, 1, 1), (1, 1, n)):
        seg = S.VoxelSegmenter(torch.from_numpy(rgb.reshape(*shape, 3)).cuda(),
                               torch.from_numpy(con.reshape(shape)).cuda(), n // 9)
        seg.iterate(4)
        out.append(seg.get_state())
        seg.close()
    a, b = out
    assert np.array_equal(a["labels"].ravel(), b["labels"].ravel())
    assert np.array_equal(a["n"], b["n"]) and np.array_equal(a["color"], b["color"])
    assert np.array_equal(a["st"], b["sx"]) and np.array_equal(a["endpoint"], b["endpoint"][:, ::-1])


@pytest.mark.parametrize("H,W", [(1, 1), (5, 3), (33, 31), (64, 90), (37, 128)])
@pytest.mark.parametrize("offset,pad", [(0, 0), (1, 3), (0, 2), (4, 0), (2, 4)])
def test_prior_output_alignment(S, H, W, offset, pad):
    import torch

    rgb, _, _ = synth.small_image(H, W, seed=H + W, n_cells=4)
    d_rgb = torch.from_numpy(rgb).cuda()
    dense = S.gradient_prior(d_rgb).cpu().numpy()
    stride = W + offset + pad
    base = torch.full((H, stride), -1.0, device="cuda")
    S.gradient_prior(d_rgb, out=base[:, offset:offset + W])
    got = base.cpu().numpy()
    assert np.array_equal(got[:, offset:offset + W], dense)
    got[:, offset:offset + W] = -1.0
    assert np.all(got == -1.0)


# one maximum per tile of 32 x 32 up to 8,192 tiles and where the workspace has
# the room, else a cleared word: the same bits (2,041 and 257 words a CTA and
# less than one each; one tile over the limit)
@pytest.mark.parametrize("H,W", [(1, 1), (65, 130), (512, 514), (1080, 1921), (2048, 4096), (2048, 4097)])
def test_prior_maximum_forms(S, H, W):
    import ctypes

    import torch

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
    assert rc == S.SCALP_OK and torch.equal(a, b)
    assert float(a.max()) == (1.0 if H * W > 1 else 0.0)


# the same limit in two dimensions, against a batch of one (lists of their own):
# 128 x 94, 191 x 63, 1117 x 11 (12,287, which once did not launch) tiles
@pytest.mark.parametrize("H,W", [(4096, 3008), (6112, 2016), (352, 35744)])
def test_list_limit(S, H, W):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(H)
    rgb = torch.randint(0, 256, (H // 16 + 1, W // 16 + 1, 3), generator=gen, dtype=torch.uint8, device="cuda")
    rgb = rgb.repeat_interleave(16, 0).repeat_interleave(16, 1)[:H, :W].contiguous()
    K = H * W // 800
    seg = S.Segmenter(rgb, None, K)
    seg.iterate(2)
    a = seg.get_state()
    seg.close()
    b = S.Batch([rgb], None, [K])
    b.iterate(2)
    g = b.get_state(0)
    b.close()
    for k in ("labels", "n", "sx", "sy", "color", "endpoint"):
        assert np.array_equal(a[k], g[k]), k
