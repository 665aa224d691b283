// scalp_phases.cuh -- the device bodies of one iteration's cluster update,
// projection (Eq. 4) and candidate lists, shared by the per-kernel launches
// (scalp_kernels.cu) and the persistent batched kernel (scalp_persistent.cu).
#pragma once

#include <cfloat>
#include <climits>

#include "scalp_internal.cuh"

namespace scalp {

// ---------------------------------------------------------------------------
// Windows.  Pixel p is a candidate of cluster k iff |x_p - x_k| <= r and
// |y_p - y_k| <= r (the (2r+1)x(2r+1) window of Algorithm 1), i.e.
// K*(n*x_p - Sx)^2 <= N*n^2 and likewise for y, evaluated exactly; each
// window becomes an inclusive integer range clipped to the image.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool in_window(long long v, long long n, long long s, long long N,
                                          long long K)
{
    __int128 d = (__int128)n * v - s;
    unsigned __int128 lhs = (unsigned __int128)K * (unsigned __int128)(d * d);
    unsigned __int128 rhs = (unsigned __int128)N * (unsigned __int128)n * (unsigned __int128)n;
    return lhs <= rhs;
}

// One end of a window, unclipped: the first (up) or last place inside, from a
// start at most a few places outside; false when the search finds none.  The
// places tried lie within r + 3 of s / n, so 64 bits hold both sides when
// they hold them at that distance (small clusters: no 128-bit products).
__device__ inline bool window_end(long long n, long long s, long long N, long long K, double r, int limit, bool up,
                                  long long &end)
{
    long long lo, hi;
    window_start(s, n, r, limit, lo, hi);
    long long v = up ? lo : hi;
    const int step = up ? 1 : -1;
    const float reach = (float)n * ((float)r + 68.0f);  // (64 further places at most)
    bool in;
    int guard = 0;
    if ((float)K * reach * reach < 9.0e18f && (float)N * (float)n * (float)n < 9.0e18f) {
        const unsigned long long rhs = (unsigned long long)N * (unsigned long long)n * (unsigned long long)n;
        do {
            const long long d = n * v - s;
            in = (unsigned long long)K * (unsigned long long)(d * d) <= rhs;
            if (!in) v += step;
        } while (!in && ++guard <= 64);
    } else {
        do {
            in = in_window(v, n, s, N, K);
            if (!in) v += step;
        } while (!in && ++guard <= 64);
    }
    end = v;
    return in;
}

__device__ __forceinline__ bool window_range(long long n, long long s, long long N, long long K, double r, int limit,
                                             int &lo, int &hi)
{
    long long l, h;
    if (!window_end(n, s, N, K, r, limit, true, l) || !window_end(n, s, N, K, r, limit, false, h)) return false;
    lo = (int)max(0LL, l);
    hi = (int)min((long long)limit - 1, h);
    return true;
}

// ---------------------------------------------------------------------------
// Projection, Eq. 4: X_k^* = argmin over p in S_k of ||X_p - X_k||, compared
// exactly as (n*x - Sx)^2 + (n*y - Sy)^2 in integers (64-bit when the image
// size bounds them below 2^62, else 128-bit), ties to the smallest raster
// index.  Searches issue PROJ_BATCH label loads per thread before comparing
// them.
// ---------------------------------------------------------------------------
constexpr int PROJ_THREADS = 512;
constexpr int PROJ_BATCH = 8;

struct ProjBest {
    unsigned long long hi, lo;
    long long p;
};

__device__ __forceinline__ bool proj_less(const ProjBest &u, const ProjBest &v)
{
    return u.hi < v.hi || (u.hi == v.hi && (u.lo < v.lo || (u.lo == v.lo && u.p < v.p)));
}

__device__ __forceinline__ void proj_shfl_min(ProjBest &b)
{
    for (int o = 16; o > 0; o >>= 1) {
        ProjBest c;
        c.hi = __shfl_xor_sync(0xffffffffu, b.hi, o);
        c.lo = __shfl_xor_sync(0xffffffffu, b.lo, o);
        c.p = __shfl_xor_sync(0xffffffffu, b.p, o);
        if (proj_less(c, b)) b = c;
    }
}



// Candidate p (raster index, pixel (x, y)) for X_k^* of cluster (n, sx, sy).
__device__ __forceinline__ ProjBest proj_candidate(long long p, int x, int y, long long n,
                                                   long long sx, long long sy, bool small)
{
    ProjBest c;
    c.p = p;
    if (small) {
        const long long dx = n * x - sx, dy = n * y - sy;
        c.hi = 0;
        c.lo = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy);
    } else {
        const __int128 dx = (__int128)n * x - sx, dy = (__int128)n * y - sy;
        const unsigned __int128 d2 = (unsigned __int128)(dx * dx) + (unsigned __int128)(dy * dy);
        c.hi = (unsigned long long)(d2 >> 64);
        c.lo = (unsigned long long)d2;
    }
    return c;
}

// ---------------------------------------------------------------------------
// Cluster update (Algorithm 1) and everything derived from it.  With
// from_acc: the means over S_k from the integer sums (an empty cluster keeps
// its colour, barycenter and endpoint), the endpoint X_k rounded half-up, and
// a projection request (Eq. 4) when the pixel there is not labelled k; the
// sums are cleared for the next assignment.  Then, from the state: the window,
// the cluster record the assignment reads, and the count of each tile the
// window overlaps (for the candidate lists).  The window the last assignment
// used is kept for the projection search.
//
// Two forms with the same results.  Up to UPDATE_LANES_MAX clusters a launch
// is bound by its chain of dependent steps, and eight lanes take a cluster:
// on one thread the five FP64 divisions (slow on this part), two 64-bit
// divisions and four window searches come one after the other (8.4 and 8.6
// us a launch for 60 and 2000 clusters, 5.4 and 6.5 on eight lanes).  Above
// it the chip is full and the extra warps only cost (120,000 clusters of a
// batch: 39.6 us on one thread each, 84.6 on eight lanes).  An iteration of
// 1080 x 1920 by lanes and by threads: 2,040 clusters 100.1 and 101.0 us, 11,972
// 101.3 and 103.0, 16,055 106.8 and 108.8, 24,012 114.2 and 114.2, 32,026 121.4
// and 118.8, 64,030 162.0 and 156.4; of two images half as high 24,012 129.3 and
// 132.0, 32,026 139.3 and 138.3.
// ---------------------------------------------------------------------------
constexpr int UPDATE_LANES = 8, UPDATE_LANES_MAX = 24576;

// One thread per cluster.
__device__ __forceinline__ void update_cluster(const SolveArgs &a, int k, int from_acc)
{
    // every load that does not depend on another is issued first: the
    // previous window, the state (kept when the cluster received no pixel)
    // and the sums; the new state then stays in registers
    const ClusterDev old = a.cdev[k];
    long long n = a.st_n[k], sx = a.st_sx[k], sy = a.st_sy[k];
    float4 col = a.st_col[k];
    int2 e = a.st_end[k];
    bool check_projection = false;
    int label_at_end = k;
    if (from_acc && k == 0) {
        // the projection searches the orphans of the assignment just finished
        // region; the count starts again for the next assignment
        a.ctr->proj_orphans = atomicExch(&a.ctr->orphans, 0);
    }
    if (from_acc) {
        const ClusterAcc c = a.acc[k];
        a.acc[k] = ClusterAcc{};
        if (c.n > 0) {
            n = (long long)c.n;
            sx = (long long)c.sx;
            sy = (long long)c.sy;
            a.st_n[k] = n;
            a.st_sx[k] = sx;
            a.st_sy[k] = sy;
            const double den = (double)n * (double)(1 << COLOR_FRAC_BITS);
            col = make_float4((float)((double)(long long)c.sL / den), (float)((double)(long long)c.sa / den),
                              (float)((double)(long long)c.sb / den), 0.f);
            a.st_col[k] = col;
            e = make_int2((int)((2 * sx + n) / (2 * n)), (int)((2 * sy + n) / (2 * n)));
            a.st_end[k] = e;
            // Eq. 4 is needed when the endpoint's pixel is not in S_k; the
            // label is read now and used last
            label_at_end = a.labels[(long long)e.y * a.W + e.x];
            check_projection = true;
        }
    }
    a.prev_win[k] = make_int4(old.xlo, old.xhi, old.ylo, old.yhi);
    ClusterDev cd;
    cd.L = col.x; cd.a = col.y; cd.b = col.z;
    cd.xk = (float)((double)sx / (double)n);
    cd.yk = (float)((double)sy / (double)n);
    cd.ex = e.x; cd.ey = e.y;
    cd.pad = k;
    const bool ok = window_range(n, sx, a.N, a.K, a.r, a.W, cd.xlo, cd.xhi) &&
                    window_range(n, sy, a.N, a.K, a.r, a.H, cd.ylo, cd.yhi);
    if (!ok) {
        atomicExch(&a.ctr->error, ERR_BAD_LABEL);
        cd.xlo = 1; cd.xhi = 0; cd.ylo = 1; cd.yhi = 0;
    }
    a.cdev[k] = cd;
    if (ok) {
        for (int ty = cd.ylo >> a.tile_shift; ty <= cd.yhi >> a.tile_shift; ++ty)
            for (int tx = cd.xlo >> a.tile_shift; tx <= cd.xhi >> a.tile_shift; ++tx)
                atomicAdd(&a.tile_count[ty * a.n_tx + tx], 1);
    }
    if (check_projection && label_at_end != k) {
        const int slot = atomicAdd(&a.ctr->nproj, 1);
        a.proj_list[slot] = k;
    }
}

// Eight lanes per cluster.  Lane i holds word i of the sums (n, Sx, Sy, SL,
// Sa, Sb), so lanes 1-5 divide side by side; lanes 0-3 search one end of the
// window each; the tiles' counts and the record's stores are spread over the
// eight.  Called by whole warps; lanes of a cluster past the last pass valid =
// false.
__device__ __forceinline__ void update_cluster_lanes(const SolveArgs &a, int k, bool valid, int from_acc)
{
    const unsigned FULL = 0xffffffffu;
    const int j = (int)(threadIdx.x % UPDATE_LANES);
    const auto from = [&](auto v, int lane) { return __shfl_sync(FULL, v, lane, UPDATE_LANES); };
    // every load that does not depend on another is issued first
    ClusterDev old{};
    long long n = 1, sx = 0, sy = 0, word = 0;
    float4 col{};
    int2 e{};
    if (valid) {
        old = a.cdev[k];
        n = a.st_n[k];
        sx = a.st_sx[k];
        sy = a.st_sy[k];
        col = a.st_col[k];
        e = a.st_end[k];
        if (from_acc) {
            static_assert(sizeof(ClusterAcc) == UPDATE_LANES * 8, "one word per lane");
            unsigned long long *acc = &a.acc[k].n + j;
            word = (long long)*acc;
            *acc = 0ull;
        }
    }
    if (from_acc && valid && k == 0 && j == 0) {
        // the projection searches the orphans of the assignment just finished
        a.ctr->proj_orphans = atomicExch(&a.ctr->orphans, 0);
    }
    const long long n_new = from(word, 0);
    const bool fresh = n_new > 0;  // (never without from_acc)
    if (fresh) n = n_new;
    {
        const long long tx = from(word, 1), ty = from(word, 2);
        if (fresh) {
            sx = tx;
            sy = ty;
        }
    }
    // lane 1, 2: Sx / n, Sy / n; lanes 3-5: the mean colour
    float mean = 0.0f;
    if (j >= 1 && j <= 5) {
        const long long num = j == 1 ? sx : j == 2 ? sy : word;
        const double den = j <= 2 ? (double)n : (double)n * (double)(1 << COLOR_FRAC_BITS);
        mean = (float)((double)num / den);
    }
    const float xk = from(mean, 1), yk = from(mean, 2), mL = from(mean, 3), ma = from(mean, 4), mb = from(mean, 5);
    if (fresh) col = make_float4(mL, ma, mb, 0.f);
    // even lanes x, odd lanes y: the endpoint, and one end of the window
    // (lanes 0, 1 the lower, 2, 3 the upper)
    const long long s = j & 1 ? sy : sx;
    int end = 0, edge = 0;
    bool ok = true;
    if (j < 4) {
        const unsigned long long num = 2ull * (unsigned long long)s + (unsigned long long)n, den = 2ull * (unsigned long long)n;
        end = (int)((num | den) >> 32 ? num / den : (unsigned long long)((unsigned)num / (unsigned)den));
        const int limit = j & 1 ? a.H : a.W;
        long long v;
        ok = window_end(n, s, a.N, a.K, a.r, limit, j < 2, v);
        edge = (int)(j < 2 ? max(0LL, v) : min((long long)limit - 1, v));
    }
    const int ex = from(end, 0), ey = from(end, 1);
    ok = from((int)ok, 0) & from((int)ok, 1) & from((int)ok, 2) & from((int)ok, 3);
    ClusterDev cd;
    cd.xlo = from(edge, 0); cd.ylo = from(edge, 1); cd.xhi = from(edge, 2); cd.yhi = from(edge, 3);
    __syncwarp();  // the cluster's old state is read before its lanes write the new one
    if (!valid) return;
    int label_at_end = k;
    if (fresh) {
        e = make_int2(ex, ey);
        // Eq. 4 is needed when the endpoint's pixel is not in S_k; the label
        // is read now and used last
        if (j == 0) label_at_end = a.labels[(long long)e.y * a.W + e.x];
    }
    if (!ok) {
        if (j == 0) atomicExch(&a.ctr->error, ERR_BAD_LABEL);
        cd.xlo = 1; cd.xhi = 0; cd.ylo = 1; cd.yhi = 0;
    }
    cd.L = col.x; cd.a = col.y; cd.b = col.z;
    cd.xk = xk; cd.yk = yk;
    cd.ex = e.x; cd.ey = e.y;
    cd.pad = k;
    if (ok) {
        // the window's tiles, one per lane in turn (a window seldom has more
        // than one or two per lane)
        const int tx0 = cd.xlo >> a.tile_shift, ty0 = cd.ylo >> a.tile_shift;
        const int nx = (cd.xhi >> a.tile_shift) - tx0 + 1, nt = nx * ((cd.yhi >> a.tile_shift) - ty0 + 1);
        for (int t = j; t < nt; t += UPDATE_LANES)
            atomicAdd(&a.tile_count[(ty0 + t / nx) * a.n_tx + tx0 + t % nx], 1);
    }
    int4 *rec = reinterpret_cast<int4 *>(&a.cdev[k]);
    if (j == 1) {
        rec[0] = make_int4(__float_as_int(cd.L), __float_as_int(cd.a), __float_as_int(cd.b), __float_as_int(cd.xk));
        a.prev_win[k] = make_int4(old.xlo, old.xhi, old.ylo, old.yhi);
    } else if (j == 2) {
        rec[1] = make_int4(__float_as_int(cd.yk), cd.ex, cd.ey, cd.xlo);
    } else if (j == 3) {
        rec[2] = make_int4(cd.xhi, cd.ylo, cd.yhi, cd.pad);
    } else if (fresh && j == 4) {
        a.st_n[k] = n;
        a.st_sx[k] = sx;
    } else if (fresh && j == 5) {
        a.st_sy[k] = sy;
        a.st_col[k] = col;
    } else if (fresh && j == 6) {
        a.st_end[k] = e;
    } else if (j == 0 && label_at_end != k) {
        a.proj_list[atomicAdd(&a.ctr->nproj, 1)] = k;
    }
}
static_assert(offsetof(ClusterDev, xk) == 12 && offsetof(ClusterDev, yk) == 16 && offsetof(ClusterDev, xlo) == 28 &&
                  offsetof(ClusterDev, xhi) == 32 && offsetof(ClusterDev, pad) == 44,
              "the record's three quarters");

// S_k lies in the window the last assignment used for cluster k, apart from
// the pixels that no window reached and that kept their label k.  The
// assignment lists those (there are seldom more than a few, but one was
// enough to make every search take the whole image: 0.8 ms more per HD solve
// for such inputs, 3.7 ms for the 32 x 240 x 320 video), and the searches go
// through the window and the list.  One warp alone is long about many: lists
// of more than N / 128 pixels, or 1,024, are left to whole CTAs, and above N / 4
// the image's rows in order are quicker than the list's scattered places.  One
// iteration of 1080 x 1920 with 2000 clusters and 3, 12, 25 and 90% of the
// columns in no window: 560, 1068, 1620, 1545 us; warps first, whatever the
// list, and never the whole image: 1615, 3915, 8516, 23648; the whole image
// from N / 16: 560, 1584, 1620, 1545; from N / 2: 560, 1073, 1830, 1545.
constexpr int PROJ_WARP_ORPHANS = 1024, PROJ_WARP_SHIFT = 7, PROJ_LIST_SHIFT = 2;
__device__ __forceinline__ bool proj_by_warp(const SolveArgs &a)
{
    const int orphans = a.ctr->proj_orphans;
    return orphans <= PROJ_WARP_ORPHANS && orphans <= a.N >> PROJ_WARP_SHIFT;
}

// The listed orphans' candidates for cluster k; thread t of `threads`.
__device__ __forceinline__ void project_orphans(const SolveArgs &a, int k, long long n, long long sx, long long sy,
                                                bool small, int t, int threads, ProjBest &b)
{
    const int count = a.ctr->proj_orphans;
    for (int i = t; i < count; i += threads) {
        const int p = a.orphan_list[i];
        if (a.labels[p] != k) continue;
        const int y = p / a.W;
        const ProjBest c = proj_candidate(p, p - y * a.W, y, n, sx, sy, small);
        if (proj_less(c, b)) b = c;
    }
}

// X_k^* is seldom far from X_k: first a warp looks at a block around the
// endpoint, 32 columns by 8 rows (one load per lane and row), then 32 by 32.
// The search is over when the block holds the argmin for certain: its best
// squared distance is below that of every pixel of the window outside it.  b
// receives the block's best (in every lane); false: the whole window has to
// be searched.  With `small` only (64-bit squared distances).
__device__ __forceinline__ bool project_near(const SolveArgs &a, int k, long long n, long long sx, long long sy,
                                             int4 win, ProjBest &b)
{
    const int lane = threadIdx.x & 31;
    const int2 e = a.st_end[k];  // X_k rounded half-up (a queued cluster's endpoint)
    const int x = e.x - 16 + lane;
    const bool in_x = x >= win.x && x <= win.y;
    const auto rows = [&](int y0) {  // the block's rows y0 .. y0 + 7
        unsigned match = 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int y = y0 + u;
            const bool in = in_x && y >= win.z && y <= win.w;
            if ((in ? a.labels[(long long)y * a.W + x] : -1) == k) match |= 1u << u;
        }
        for (; match; match &= match - 1) {
            const int y = y0 + __ffs(match) - 1;
            const ProjBest c = proj_candidate((long long)y * a.W + x, x, y, n, sx, sy, true);
            if (proj_less(c, b)) b = c;
        }
    };
    // the least squared distance outside columns e.x - 16 .. e.x + 15 and rows
    // ylo .. yhi (none where the window ends inside)
    const auto outside = [&](int ylo, int yhi) {
        long long d = LLONG_MAX;
        if (win.x < e.x - 16) d = min(d, sx - n * (e.x - 17));
        if (win.y > e.x + 15) d = min(d, n * (e.x + 16) - sx);
        if (win.z < ylo) d = min(d, sy - n * (ylo - 1));
        if (win.w > yhi) d = min(d, n * (yhi + 1) - sy);
        return d == LLONG_MAX ? ~0ull : (unsigned long long)(d * d);
    };
    rows(e.y - 4);
    proj_shfl_min(b);
    if (b.p != LLONG_MAX && b.lo < outside(e.y - 4, e.y + 3)) return true;
#pragma unroll 1
    for (int y0 = e.y - 12; y0 <= e.y + 12; y0 += 8)
        if (y0 != e.y - 4) rows(y0);
    proj_shfl_min(b);
    return b.p != LLONG_MAX && b.lo < outside(e.y - 12, e.y + 19);
}

// X_k^* of cluster k, by one lane.
__device__ __forceinline__ void project_store(const SolveArgs &a, int k, const ProjBest &b)
{
    if (b.p == LLONG_MAX) {
        atomicExch(&a.ctr->error, ERR_BAD_LABEL);
        return;
    }
    const int p = (int)b.p, ey = p / a.W, ex = p - ey * a.W;  // (N <= 2^30)
    a.st_end[k] = make_int2(ex, ey);
    a.cdev[k].ex = ex;
    a.cdev[k].ey = ey;
}

__device__ __forceinline__ bool proj_small(const SolveArgs &a, long long n)
{
    const double bound = (double)max(a.W, a.H);
    return 2.0 * (n * bound) * (n * bound) < 4.0e18;
}

// The `end` pixels of rows of div.d pixels from (xlo, ylo) for cluster k by
// `threads` threads, of which this is thread t.  BATCH label loads are issued
// before any is compared; the matches, seldom more than a few, are then taken
// one by one.  (The kernels are short and their code is cold on every launch:
// distances written out for each load of the batch cost more in instruction
// fetches than they saved.)
template <int BATCH, bool EXACT>
__device__ __forceinline__ void project_scan_rows(const SolveArgs &a, int k, long long n, long long sx, long long sy,
                                                  bool small, int xlo, int ylo, Divisor div, unsigned end, int t,
                                                  int threads, ProjBest &b)
{
    // (not __restrict__: the persistent kernel writes the labels between its
    // barriers, so no load of theirs may take the read-only path)
    const int *corner = a.labels + (long long)ylo * a.W + xlo;
    for (unsigned base = (unsigned)t; base < end; base += (unsigned)(threads * BATCH)) {
        unsigned match = 0u;
        int lab[BATCH], row, col;
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            // (past the end: the last pixel, which changes nothing)
            div.split<EXACT>(min(base + (unsigned)(u * threads), end - 1u), row, col);
            lab[u] = corner[row * a.W + col];
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) match |= lab[u] == k ? 1u << u : 0u;
        for (; match; match &= match - 1) {
            div.split<EXACT>(min(base + (unsigned)((__ffs(match) - 1) * threads), end - 1u), row, col);
            const int x = xlo + col, y = ylo + row;
            const ProjBest c = proj_candidate((long long)y * a.W + x, x, y, n, sx, sy, EXACT || small);
            if (proj_less(c, b)) b = c;
        }
    }
}

// The w x h pixels from (xlo, ylo).  Windows below 1,626 x 1,626 divide
// exactly and their clusters have 64-bit squared distances; larger ones and
// those of large clusters take the general form, with as many loads in flight
// (one at a time, solves of 2160 x 3840 with 12 clusters took 34.8 ms per two
// iterations against 31.4).
template <int BATCH>
__device__ __forceinline__ void project_scan(const SolveArgs &a, int k, long long n, long long sx, long long sy,
                                             bool small, int xlo, int ylo, int w, int h, int t, int threads,
                                             ProjBest &b)
{
    const Divisor div((unsigned)max(w, 1));
    const unsigned end = (unsigned)(max(w, 0) * max(h, 0));  // (within the image: at most 2^30)
    if (small && div.exact(end)) project_scan_rows<BATCH, true>(a, k, n, sx, sy, small, xlo, ylo, div, end, t, threads, b);
    else project_scan_rows<BATCH, false>(a, k, n, sx, sy, small, xlo, ylo, div, end, t, threads, b);
}

// Eq. 4 for queued cluster j of one image by one warp: the same argmin, with
// the same exact comparison and tie rule, as the CTA-wide search.
__device__ __forceinline__ void project_warp(const SolveArgs &a, int j)
{
    const int lane = threadIdx.x & 31;
    const int k = a.proj_list[j];
    const long long n = a.st_n[k], sx = a.st_sx[k], sy = a.st_sy[k];
    const int4 w4 = a.prev_win[k];
    const bool small = proj_small(a, n);
    ProjBest b = {~0ull, ~0ull, LLONG_MAX};
    if (!small || !project_near(a, k, n, sx, sy, w4, b)) {
        project_scan<4>(a, k, n, sx, sy, small, w4.x, w4.z, w4.y - w4.x + 1, w4.w - w4.z + 1, lane, 32, b);
    }
    project_orphans(a, k, n, sx, sy, small, lane, 32, b);
    proj_shfl_min(b);
    if (lane == 0) project_store(a, k, b);
}

// Queued projections over the window and the orphans (with whole_image, at
// set-up, or very many orphans the whole image).  Queue entries j0, j0 + stride,
// ... of one image.  Each warp first looks near the endpoint of one (as many at a time as the CTA
// has warps), and only what it cannot settle there the whole CTA searches,
// cluster by cluster.  Per launch, against a CTA per cluster over its whole
// window: HD 10.7 -> 9.5 us, UHD 20.6 -> 13.1.
__device__ __forceinline__ void project_cta(const SolveArgs &a, int whole_image, int j0, int stride)
{
    constexpr int WARPS = PROJ_THREADS / 32;
    __shared__ ProjBest s_best[WARPS];
    __shared__ int s_left[WARPS];  // per warp: the cluster left to the CTA, or -1
    const int nproj = a.ctr->nproj;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool look = !whole_image && proj_by_warp(a);
    const bool whole = whole_image || a.ctr->proj_orphans > a.N >> PROJ_LIST_SHIFT;
    for (long long first = j0; first < nproj; first += (long long)stride * WARPS) {
        if (look) {
            const long long j = first + (long long)stride * warp;
            int left = -1;
            if (j < nproj) {
                const int k = a.proj_list[j];
                const long long n = a.st_n[k], sx = a.st_sx[k], sy = a.st_sy[k];
                ProjBest b = {~0ull, ~0ull, LLONG_MAX};
                left = k;
                if (proj_small(a, n) && project_near(a, k, n, sx, sy, a.prev_win[k], b)) {
                    project_orphans(a, k, n, sx, sy, true, lane, 32, b);
                    proj_shfl_min(b);
                    if (lane == 0) project_store(a, k, b);
                    left = -1;
                }
            }
            if (lane == 0) s_left[warp] = left;
            __syncthreads();
        }
#pragma unroll 1
        for (int q = 0; q < WARPS; ++q) {
            const long long j = first + (long long)stride * q;
            if (j >= nproj) break;
            const int k = look ? s_left[q] : a.proj_list[j];
            if (k < 0) continue;
            const long long n = a.st_n[k], sx = a.st_sx[k], sy = a.st_sy[k];
            int xlo = 0, xhi = a.W - 1, ylo = 0, yhi = a.H - 1;
            if (!whole) {
                const int4 w4 = a.prev_win[k];
                xlo = w4.x; xhi = w4.y; ylo = w4.z; yhi = w4.w;
            }
            const bool small = proj_small(a, n);
            ProjBest b = {~0ull, ~0ull, LLONG_MAX};
            project_scan<PROJ_BATCH>(a, k, n, sx, sy, small, xlo, ylo, xhi - xlo + 1, yhi - ylo + 1, tid, PROJ_THREADS,
                                     b);
            if (!whole) project_orphans(a, k, n, sx, sy, small, tid, PROJ_THREADS, b);
            proj_shfl_min(b);
            if (lane == 0) s_best[warp] = b;
            __syncthreads();
            if (warp == 0) {
                b = lane < WARPS ? s_best[lane] : ProjBest{~0ull, ~0ull, LLONG_MAX};
                proj_shfl_min(b);
                if (lane == 0) project_store(a, k, b);
            }
            __syncthreads();
        }
        if (look) __syncthreads();  // s_left is written again
    }
}

// ---------------------------------------------------------------------------
// Per-tile candidate lists: exclusive scan of the tile counts, then one thread
// per (cluster, tile) slot files the cluster into each tile its window
// overlaps, at tile_off[t] + (a per-tile cursor).  The assignment CTA of tile
// t zeroes tile_count[t] and tile_cursor[t] once it has read its list (set-up
// and set_state zero them on the host side).  The lists touch no other
// counter, so they can run beside the projection: the update restarts the
// orphan count and the assignment the projection queue.
// ---------------------------------------------------------------------------

// tile_off from the counts and the overflow check.
__device__ __forceinline__ void publish_offsets(const SolveArgs &a, const int *off)
{
    const int n = a.n_tx * a.n_ty;
    for (int i = threadIdx.x; i <= n; i += blockDim.x) a.tile_off[i] = off[i];
    if (threadIdx.x == 0 && off[n] > a.tile_cap) atomicExch(&a.ctr->error, ERR_TILE_LIST_OVERFLOW);
}

constexpr int SCAN1_THREADS = 1024;

// tile_off of one image by one CTA of THREADS threads.
template <int THREADS = SCAN1_THREADS>
__device__ __forceinline__ void scan_tiles_cta(const SolveArgs &a)
{
    __shared__ int s_warp[32];
    cta_scan(a.tile_count, a.tile_off, a.n_tx * a.n_ty, THREADS, s_warp);
    if (threadIdx.x == 0) {
        const int n = a.n_tx * a.n_ty;
        if (a.tile_off[n] > a.tile_cap) atomicExch(&a.ctr->error, ERR_TILE_LIST_OVERFLOW);
    }
}

__device__ __forceinline__ void fill_slot(const SolveArgs &a, long long i)
{
    const long long slots = (long long)a.tpw_x * a.tpw_y;
    if (i >= (long long)a.Keff * slots) return;
    const int k = (int)(i / slots), j = (int)(i % slots);
    const ClusterDev cd = a.cdev[k];
    if (cd.xlo > cd.xhi) return;
    const int tx = (cd.xlo >> a.tile_shift) + j % a.tpw_x, ty = (cd.ylo >> a.tile_shift) + j / a.tpw_x;
    if (tx > cd.xhi >> a.tile_shift || ty > cd.yhi >> a.tile_shift) return;
    const int t = ty * a.n_tx + tx;
    const int pos = a.tile_off[t] + atomicAdd(&a.tile_cursor[t], 1);
    if (pos < a.tile_cap) a.tile_list[pos] = k;
}

}  // namespace scalp
