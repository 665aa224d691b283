"""Index arithmetic of the kernels at the limits of the accepted sizes (H * W <=
2^30), from the header that they include, compiled for the host.  Places on the
plane that the distance maps' build reads: a warp covers rows past the box's
last one; the places formed for them stay inside the box.  Rows and columns of
the projections' windows: the divisions by a reciprocal are exact."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_1903_07149_gb300", "csrc", "scalp_offsets.h")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("offsets")
    src, so = d / "offsets.cpp", d / "offsets.so"
    src.write_text(f'#include "{HEADER}"\n'
                   'extern "C" int rows_per_pass() { return 4 * scalp::STRIP_ROWS; }\n'
                   'extern "C" void places(int lrow, int rows, int pitch, int width, int col, unsigned *o)\n'
                   "{ const scalp::StripPlaces s = scalp::strip_places(lrow, rows, pitch, width, col);\n"
                   "  o[0] = s.off; o[1] = s.step; o[2] = s.last; o[3] = s.end; o[4] = s.more; }\n")
    src.write_text(src.read_text() +
                   'extern "C" int exact(unsigned d, unsigned end) { return scalp::Divisor(d).exact(end); }\n'
                   'extern "C" void split(unsigned d, int ex, const unsigned *i, int n, int *q, int *r)\n'
                   "{ const scalp::Divisor v(d);\n"
                   "  for (int j = 0; j < n; ++j) {\n"
                   "    if (ex) v.split<true>(i[j], q[j], r[j]); else v.split<false>(i[j], q[j], r[j]); } }\n")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


LIMIT = 1 << 30
# widths around 2^31 / 15 (where fifteen rows leave 31 bits), 2^32 / 15 and 2^28
# (where four rows leave 30), and the widest image of each height
WIDTHS = [143165575, 143165576, 143165580, 150000000, 200000000, (1 << 28) - 1, 1 << 28, (1 << 28) + 1,
          286331148, 286331156, LIMIT]


@pytest.mark.parametrize("H", [1, 2, 3, 4, 5, 6, 7, 8, 15, 16, 17, 31, 32, 33, 4095])
def test_places_stay_in_the_box(lib, H):
    o = (ctypes.c_uint * 5)()
    per_pass = lib.rows_per_pass()
    for W in sorted({w for w in WIDTHS if w * H <= LIMIT} | {LIMIT // H}):
        pitch = (W + 3) & ~3
        for rows in sorted({1, H, (H + 1) // 2}):
            for width, col in ((W, 0), (W, W - 1), (1, 0), (1, 7), (5, 4), (5, 6)):
                c = min(col, width - 1)
                for lrow in range(4):
                    lib.places(lrow, rows, pitch, width, col, o)
                    place, step, last, end, more = o
                    stored = {}  # by the map row that the lane writes
                    for i in range(-(-rows // per_pass) * per_pass // 4):
                        assert place == (lrow + (4 * i if step else 0)) * pitch + c < 1 << 32  # (nothing wrapped)
                        read = min(place, last)
                        assert read <= (rows - 1) * pitch + width - 1
                        if place < (end if i % (per_pass // 4) == 0 else more):
                            stored[lrow + 4 * i] = read
                        place += step
                    assert place < 1 << 32
                    assert stored == ({row: row * pitch + c for row in range(lrow, rows, 4)} if col < width else {})


def test_divisions_are_exact(lib):
    rng = np.random.default_rng(11)
    widths = list(range(1, 70)) + [481, 1080, 1625, 1626, 1920, 3840, 4096, 32767, 32768, 32769, 65535, 65536, 65537,
                                   LIMIT // 3, LIMIT // 2, LIMIT - 1, LIMIT]
    widths += [int(2 ** v) for v in rng.uniform(6, 30, 300)]
    forms = set()
    for d in widths:
        for end in (d, min(LIMIT, 1625 * d), min(LIMIT, max(1, ((1 << 32) - 1) // d)), LIMIT // d * d):
            ex = lib.exact(d, ctypes.c_uint(end))
            assert bool(ex) == (d > 1 and end * d < 1 << 32)
            q0 = rng.integers(0, max(1, end // d), 40)
            i = np.concatenate([np.arange(0, min(end, 20)), rng.integers(0, end, 60), end - 1 - np.arange(min(end, 20)),
                                q0 * d, q0 * d + d - 1, np.maximum(q0 * d - 1, 0)]).astype(np.int64)
            i = np.ascontiguousarray(i[i < end], np.uint32)
            for form in {0, ex}:
                q, r = np.empty(i.size, np.int32), np.empty(i.size, np.int32)
                lib.split(d, form, ctypes.c_void_p(i.ctypes.data), i.size, ctypes.c_void_p(q.ctypes.data),
                          ctypes.c_void_p(r.ctypes.data))
                assert np.array_equal(q, i // d) and np.array_equal(r, i % d), (d, end, form)
                forms.add(form)
    assert forms == {0, 1}


# Thin images whose pitch times the rows of a warp's batch leaves 32 bits
# (fifteen rows, and four), against the paths walked on the plane without maps
@pytest.mark.gpu
@pytest.mark.parametrize("H,W", [(1, 150_000_001), (1, (1 << 28) + 5), (5, 150_000_000)])
@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_thin_images_with_maps(H, W, storage):
    import torch

    from paper_1903_07149_gb300 import build as scalp_build
    from paper_1903_07149_gb300 import scalp as S

    scalp_build.build()
    gen = torch.Generator(device="cuda").manual_seed(W)
    cells = torch.randint(0, 256, (1, W // 40 + 1, 3), generator=gen, dtype=torch.uint8, device="cuda")
    rgb = cells.repeat_interleave(40, 1)[:, :W].expand(H, W, 3).contiguous()
    rgb[:, ::7] ^= 21
    K = W // 100
    labels = []
    for global_walk in (False, True):
        seg = S.Segmenter(rgb, None, K, storage=storage, global_walk=global_walk)
        seg.iterate(2)
        out = torch.empty((H, W), dtype=torch.int32, device="cuda")
        seg.labels(enforce=False, out=out)
        labels.append(out)
        if not global_walk:
            seg.count_samples(1)
            seg.iterate(1)
            assert seg.count_samples(0, rects=True)[2] > 0  # maps were used
        seg.close()
        del seg
        torch.cuda.empty_cache()
    assert torch.equal(*labels)
