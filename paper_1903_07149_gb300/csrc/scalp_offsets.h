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

// Division of i < 2^30 by d >= 1 through rcp = ceil(2^32 / d): i * rcp / 2^32
// exceeds i / d by less than i / 2^32 < 1/4, so its floor is the quotient or
// one more, and then the remainder is negative.  For all i <= end with end * d
// < 2^32 (and d > 1) the excess is below 1 / d and the floor is the quotient:
// EXACT leaves the correction out.
struct Divisor {
    unsigned d, rcp;

    SCALP_HD explicit Divisor(unsigned d_) : d(d_), rcp(d_ > 1u ? 0xffffffffu / d_ + 1u : 0u) {}
    SCALP_HD bool exact(unsigned end) const { return d > 1u && (unsigned long long)end * d < (1ull << 32); }
    template <bool EXACT>
    SCALP_HD void split(unsigned i, int &quotient, int &remainder) const
    {
        const unsigned q = EXACT || rcp ? (unsigned)((unsigned long long)i * rcp >> 32) : i;
        const int r = (int)(i - q * d);
        const bool over = !EXACT && r < 0;
        quotient = (int)q - (over ? 1 : 0);
        remainder = over ? r + (int)d : r;
    }
};

}  // namespace scalp
