// scalp_offsets.h -- index arithmetic of the kernels in plain C++, so that the
// very code they run can be compiled for the host and checked at the limits of
// its ranges.
#pragma once

#ifdef __CUDACC__
#define SCALP_HD __host__ __device__ __forceinline__
#else
#define SCALP_HD inline
#endif

namespace scalp {

// Places on the plane of one lane's column of a strip of a distance-map box:
// rows lrow, lrow + 4, ... from the box's first pixel, STRIP_ROWS of them per
// pass until all `rows` are covered.  Row i of a pass lies at
// min(off + i * step, last), off advancing by step per row; a row past the box
// takes the box's last.  A pass stores its first row where off is below end,
// and its others where theirs is below more.
//
// Rows past the box may lie outside the image, so the places before the
// minimum are unsigned 32-bit words that never wrap.  A plane has H rows of at
// most W + 3, H * W <= 2^30, and a mapped box has fewer than 2^15 of them.  A
// box of more than four rows forms places up to row 4 * STRIP_ROWS * passes
// + 3, at most 3.8 times its rows (19 for five): below 3.8 * (2^30 + 3 * 2^15)
// < 2^32.  A box of up to four rows takes step 0 and stores no more than a
// lane's first row, at most the fourth.
// (Signed words overflowed on images of up to seven rows from 143 million
// columns on, and read outside the plane.)
constexpr int STRIP_ROWS = 4;

struct StripPlaces {
    unsigned off, step, last, end, more;
};

SCALP_HD StripPlaces strip_places(int lrow, int rows, int pitch, int width, int col)
{
    const unsigned p = (unsigned)pitch, c = (unsigned)(col < width ? col : width - 1);
    StripPlaces s;
    s.off = (unsigned)lrow * p + c;
    s.step = rows > 4 ? 4u * p : 0u;
    s.last = (unsigned)(rows - 1) * p + c;
    s.end = col < width ? s.last + 1u : 0u;
    s.more = rows > 4 ? s.end : 0u;
    return s;
}

}  // namespace scalp
