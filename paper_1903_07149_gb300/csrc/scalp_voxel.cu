// scalp_voxel.cu -- supervoxels: SCALP on a video volume (T frames x H x W),
// the extension the paper's conclusion names as future work.  Each rule is the
// 2-D one taken axis by axis:
//   * r = cbrt(N/K) (computed on the host); a 3-D regular grid of step r;
//   * candidates of cluster k: |v - s_v/n| <= r on each axis, r the real
//     cube root of N/K, i.e. K*|n*v - s_v|^3 <= N*n^3 decided exactly, kept
//     as integer bounds per axis;
//   * the linear path is a 3-D digital segment traced from the
//     lexicographically smaller end (x, then y, then t); the axis with the
//     largest |delta| (ties: x, y, t) steps by one, each other axis by
//     round-half-up(i*|delta_j|/ns);
//   * D is Eq. 3 with the squared 3-D distance, the colour and contour terms of
//     Eq. 1-2 along the path;
//   * update and projection (Eq. 4) as in 2-D, with the voxel index as the
//     tie-break; there is no connectivity step.
//
// One iteration is three kernels: assignment (one 512-thread CTA per 16x8x4
// tile, one voxel per thread, paths walked in global memory, warp-aggregated
// integer sums), update (eight lanes per cluster), and one launch for the
// candidate lists (count scan and slot fill) and the projection (one CTA per
// queued cluster).
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "scalp_launch.h"
#include "../../include/scalp.h"

namespace scalp {
namespace {

constexpr int VTX = 16, VTY = 8, VTT = 4;  // voxel tile
constexpr int VTILE = VTX * VTY * VTT;     // 512 voxels, one per thread
constexpr int VPROJ_THREADS = 512;

struct VoxCluster {  // 64 bytes: what the assignment reads about cluster k
    float L, a, b;
    float xk, yk, tk;
    int ex, ey, et;
    int xlo, xhi, ylo, yhi, tlo, thi;
    int pad;
};
static_assert(sizeof(VoxCluster) == 64, "VoxCluster layout");

struct VoxAcc {  // 64 bytes: integer sums of one assignment
    unsigned long long n, sx, sy, st, sL, sa, sb, pad;
};

struct VoxArgs {
    int T, H, W, K, Keff, nx, ny, nt;
    long long N, HW;
    double r;
    float lam, gamma, ms2;
    int n_tx, n_ty, n_tt;
    int tpw_x, tpw_y, tpw_t;  // bound on the tiles one window spans, per axis
    long long tile_cap;
    int count_samples;
    int thin_w, thin_h, thin_d;  // voxels of a tile along each axis, where the volume is thinner than it
    const float4 *plane;      // (L, a, b, w) per voxel
    int *labels;
    long long *st_n, *st_sx, *st_sy, *st_st;
    float4 *st_col;
    int4 *st_end;             // (ex, ey, et, 0)
    VoxCluster *cdev;
    VoxAcc *acc;
    int *prev_win;            // 6 ints per cluster: the window the last assignment used
    int *proj_list;
    int *orphan_list;         // voxel indices of the last assignment's orphans (room for N)
    int *tile_count, *tile_off, *tile_cursor, *tile_list;
    DevCounters *ctr;
    const float *lut;
};

// ---------------------------------------------------------------------------
// Windows: |v - s/n| <= r with r^3 = N/K, i.e. K*q^3 <= N*n^3 for
// q = |n*v - s|.  An FP32 comparison of q/n with r (each within 4e-7
// relative of exact) decides every value farther than 1e-5 relative from the
// edge; the rest are decided in 128-bit integers.  There q <= (1 + 1e-5) n r,
// and a volume holds at most 2^30 voxels (n, N <= 2^30), so K*q^3 and N*n^3
// both stay below 2^121.
// ---------------------------------------------------------------------------
__device__ __forceinline__ bool vin_window(long long v, long long n, long long s, long long N, long long K,
                                           double r)
{
    const long long d = n * v - s;
    const unsigned long long q = (unsigned long long)(d < 0 ? -d : d);
    // FP32 filter: q/n and r each within 4e-7 relative of exact, so outside
    // a 1e-5 band the FP32 comparison is the exact one
    const float x = __fdividef((float)q, (float)n), rf = (float)r;
    if (x < rf * (1.0f - 1e-5f)) return true;
    if (x > rf * (1.0f + 1e-5f)) return false;
    const unsigned __int128 lhs = (unsigned __int128)q * q * q * (unsigned long long)K;
    const unsigned __int128 rhs =
        (unsigned __int128)((unsigned long long)N * (unsigned long long)n) * ((unsigned long long)n * (unsigned long long)n);
    return lhs <= rhs;
}

// One end of a window clipped to [0, lim): the first (up) or last place inside
// (past the other end's start when none is: the window is empty).
__device__ __forceinline__ int vwindow_end(long long n, long long s, long long N, long long K, double r, int lim,
                                           bool up)
{
    long long lo, hi;
    window_start(s, n, r, lim, lo, hi);
    const int first = (int)max(lo, 0LL), last = (int)min(hi, (long long)lim - 1);
    int v = up ? first : last;
    const int step = up ? 1 : -1;
    while (v >= first && v <= last && !vin_window(v, n, s, N, K, r)) v += step;
    return v;
}

// ---------------------------------------------------------------------------
// Integer sums of (1, x, y, t, L, a, b) per label; colour fixed point
// 2^COLOR_FRAC_BITS.  A warp's 32 voxels lie in one tile, or share a frame and lie within 32
// columns and 2 rows of a base, so the three offsets pack into one 32-bit
// warp sum (10 bits each).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void vaggregate(const VoxArgs &a, bool valid, int lab, int bx, int by, int bt,
                                           int dx, int dy, int dt, float4 v)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const float scale = (float)(1 << COLOR_FRAC_BITS);
    const int qL = valid ? __float2int_rn(v.x * scale) : 0;
    const int qa = valid ? __float2int_rn(v.y * scale) : 0;
    const int qb = valid ? __float2int_rn(v.z * scale) : 0;
    const unsigned qc = valid ? (unsigned)dx | ((unsigned)dy << 10) | ((unsigned)dt << 20) : 0u;
    unsigned pending = __ballot_sync(FULL, valid);
    while (pending) {
        const int leader = __ffs(pending) - 1;
        const int k = __shfl_sync(FULL, lab, leader);
        const bool mine = valid && lab == k;
        const unsigned grp = __ballot_sync(FULL, mine);
        const long long cnt = __popc(grp);
        const unsigned sc = __reduce_add_sync(FULL, mine ? qc : 0u);
        const long long sL = (int)__reduce_add_sync(FULL, mine ? (unsigned)qL : 0u);
        const long long sa = (int)__reduce_add_sync(FULL, mine ? (unsigned)qa : 0u);
        const long long sb = (int)__reduce_add_sync(FULL, mine ? (unsigned)qb : 0u);
        if (lane == leader) {
            VoxAcc *c = &a.acc[k];
            atomicAdd(&c->n, (unsigned long long)cnt);
            atomicAdd(&c->sx, (unsigned long long)(cnt * bx + (long long)(sc & 0x3ffu)));
            atomicAdd(&c->sy, (unsigned long long)(cnt * by + (long long)((sc >> 10) & 0x3ffu)));
            atomicAdd(&c->st, (unsigned long long)(cnt * bt + (long long)(sc >> 20)));
            atomicAdd(&c->sL, (unsigned long long)sL);
            atomicAdd(&c->sa, (unsigned long long)sa);
            atomicAdd(&c->sb, (unsigned long long)sb);
        }
        pending &= ~grp;
    }
}

// ---------------------------------------------------------------------------
// Set-up: CIELab, contour factor, grid label, initial sums.
// ---------------------------------------------------------------------------
// One warp per 32-voxel row segment: CIELab, contour factor, plane sample
// and grid label of each voxel, then the warp-aggregated integer sums of the
// initial clusters from the values just stored (the sums start at zero).
// The frame and row come once per segment; the cell column by a 32-bit
// division when W * nx < 2^32.
__global__ void __launch_bounds__(256) k_vsetup(VoxArgs a, const uint8_t *__restrict__ rgb,
                                               const float *__restrict__ contour, float sigma, float4 *plane)
{
    __shared__ float lin[256];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) lin[i] = a.lut[i];
    __syncthreads();
    const float inv_s2 = 1.0f / (sigma * sigma);
    const long long segs_per_row = (a.W + 31) / 32;
    const long long n_segs = segs_per_row * a.H * a.T;
    const long long warps = (long long)gridDim.x * (blockDim.x / 32);
    const int lane = threadIdx.x & 31;
    const bool narrow = (unsigned long long)a.W * (unsigned long long)a.nx < (1ULL << 32);
    for (long long s = blockIdx.x * (long long)(blockDim.x / 32) + (threadIdx.x >> 5); s < n_segs; s += warps) {
        const long long row = s / segs_per_row;
        const int x0 = (int)(s - row * segs_per_row) * 32;
        const int t = (int)(row / a.H), y = (int)(row - (long long)t * a.H);
        const int x = x0 + lane;
        const bool valid = x < a.W;
        const long long p = ((long long)t * a.H + y) * a.W + x;
        const int cy = (int)((long long)y * a.ny / a.H), ct = (int)((long long)t * a.nt / a.T);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        int lab = -1;
        if (valid) {
            const float3 c3 = srgb_to_lab(lin, rgb + 3 * p);
            const float c = contour ? contour[p] : 0.0f;
            v = make_float4(c3.x, c3.y, c3.z, -expm1f(-(c * c) * inv_s2));
            plane[p] = v;
            const int cx = narrow ? (int)((unsigned)x * (unsigned)a.nx / (unsigned)a.W)
                                  : (int)((long long)x * a.nx / a.W);
            lab = (ct * a.ny + cy) * a.nx + cx;
            a.labels[p] = lab;
        }
        vaggregate(a, valid, lab, x0, y, t, lane, 0, 0, v);
    }
}

// ---------------------------------------------------------------------------
// Update: means, endpoint, projection request, window, record, tile counts.
// ---------------------------------------------------------------------------
// Eight lanes per cluster, as in 2-D (scalp_phases.cuh): lane i holds word i
// of the sums, lanes 1-6 divide side by side, lanes 0-5 search one end of the
// window each, and the stores are spread (12.3 us a launch for 2000 clusters
// on one thread each, 7.5 now).
constexpr int VUPDATE_LANES = 8, VUPDATE_THREADS = 64;

__global__ void __launch_bounds__(VUPDATE_THREADS) k_vupdate(VoxArgs a, int from_acc)
{
    pdl_wait();
    pdl_release();
    const unsigned FULL = 0xffffffffu;
    const int g = (blockIdx.x * VUPDATE_THREADS + (int)threadIdx.x) / VUPDATE_LANES;
    const int k = min(g, a.Keff - 1), j = (int)(threadIdx.x % VUPDATE_LANES);
    const bool valid = g < a.Keff;
    const auto from = [&](auto v, int lane) { return __shfl_sync(FULL, v, lane, VUPDATE_LANES); };
    const VoxCluster old = a.cdev[k];
    long long n = a.st_n[k], sx = a.st_sx[k], sy = a.st_sy[k], st = a.st_st[k], word = 0;
    float4 col = a.st_col[k];
    int4 e = a.st_end[k];
    if (from_acc && valid) {
        static_assert(sizeof(VoxAcc) == VUPDATE_LANES * 8, "one word per lane");
        unsigned long long *acc = &a.acc[k].n + j;
        word = (long long)*acc;
        *acc = 0ull;
        // the projection searches the orphans of the assignment just finished
        if (k == 0 && j == 0) a.ctr->proj_orphans = atomicExch(&a.ctr->orphans, 0);
    }
    const long long n_new = from(word, 0), nsx = from(word, 1), nsy = from(word, 2), nst = from(word, 3);
    const bool fresh = n_new > 0;  // an empty cluster keeps its state
    if (fresh) {
        n = n_new;
        sx = nsx;
        sy = nsy;
        st = nst;
    }
    const auto axis = [&](int i) { return i == 0 ? sx : i == 1 ? sy : st; };
    float mean = 0.0f;  // lanes 1-3: the barycenter, 4-6: the mean colour
    if (j >= 1 && j <= 6) {
        const double den = j <= 3 ? (double)n : (double)n * (double)(1 << COLOR_FRAC_BITS);
        mean = (float)((double)(j <= 3 ? axis(j - 1) : word) / den);
    }
    VoxCluster cd;
    cd.xk = from(mean, 1); cd.yk = from(mean, 2); cd.tk = from(mean, 3);
    const float mL = from(mean, 4), ma = from(mean, 5), mb = from(mean, 6);
    if (fresh) col = make_float4(mL, ma, mb, 0.f);
    int end = 0, edge = 0;  // axis j mod 3: the endpoint, and the lower (0-2) or upper (3-5) end of the window
    if (j < 6) {
        const int i = j % 3;
        const long long s = axis(i);
        const unsigned long long num = 2ull * (unsigned long long)s + (unsigned long long)n, den = 2ull * (unsigned long long)n;
        end = (int)((num | den) >> 32 ? num / den : (unsigned long long)((unsigned)num / (unsigned)den));
        edge = vwindow_end(n, s, a.N, a.K, a.r, i == 0 ? a.W : i == 1 ? a.H : a.T, j < 3);
    }
    const int ex = from(end, 0), ey = from(end, 1), et = from(end, 2);
    cd.xlo = from(edge, 0); cd.ylo = from(edge, 1); cd.tlo = from(edge, 2);
    cd.xhi = from(edge, 3); cd.yhi = from(edge, 4); cd.thi = from(edge, 5);
    __syncwarp();  // the cluster's old state is read before its lanes write the new one
    if (!valid) return;
    int label_at_end = k;
    if (fresh) {
        e = make_int4(ex, ey, et, 0);
        if (j == 0) label_at_end = a.labels[((long long)et * a.H + ey) * a.W + ex];
    }
    cd.L = col.x; cd.a = col.y; cd.b = col.z;
    cd.ex = e.x; cd.ey = e.y; cd.et = e.z;
    cd.pad = k;
    if (cd.xlo <= cd.xhi && cd.ylo <= cd.yhi && cd.tlo <= cd.thi) {
        const int tx0 = cd.xlo / VTX, ty0 = cd.ylo / VTY, tt0 = cd.tlo / VTT;
        const int nx = cd.xhi / VTX - tx0 + 1, ny = cd.yhi / VTY - ty0 + 1, nt = nx * ny * (cd.thi / VTT - tt0 + 1);
        for (int i = j; i < nt; i += VUPDATE_LANES) {
            const int row = i / nx, fr = row / ny;
            atomicAdd(&a.tile_count[((tt0 + fr) * a.n_ty + ty0 + row - fr * ny) * a.n_tx + tx0 + i - row * nx], 1);
        }
    }
    int4 *rec = reinterpret_cast<int4 *>(&a.cdev[k]);
    const auto fi = [](float v) { return __float_as_int(v); };
    if (j == 1) {
        rec[0] = make_int4(fi(cd.L), fi(cd.a), fi(cd.b), fi(cd.xk));
        if (fresh) a.st_col[k] = col;
    } else if (j == 2) {
        rec[1] = make_int4(fi(cd.yk), fi(cd.tk), cd.ex, cd.ey);
        if (fresh) a.st_end[k] = e;
    } else if (j == 3) {
        rec[2] = make_int4(cd.et, cd.xlo, cd.xhi, cd.ylo);
    } else if (j == 4) {
        rec[3] = make_int4(cd.yhi, cd.tlo, cd.thi, cd.pad);
    } else if (j == 5) {
        int2 *pw = reinterpret_cast<int2 *>(a.prev_win + 6 * (long long)k);
        pw[0] = make_int2(old.xlo, old.xhi);
        pw[1] = make_int2(old.ylo, old.yhi);
        pw[2] = make_int2(old.tlo, old.thi);
    } else if (fresh && j == 6) {
        a.st_n[k] = n;
        a.st_sx[k] = sx;
    } else if (fresh && j == 7) {
        a.st_sy[k] = sy;
        a.st_st[k] = st;
    } else if (j == 0 && label_at_end != k) {
        a.proj_list[atomicAdd(&a.ctr->nproj, 1)] = k;
    }
}
static_assert(offsetof(VoxCluster, yk) == 16 && offsetof(VoxCluster, ex) == 24 && offsetof(VoxCluster, et) == 32 &&
                  offsetof(VoxCluster, yhi) == 48 && offsetof(VoxCluster, pad) == 60,
              "the record's four quarters");

// ---------------------------------------------------------------------------
// Projection (Eq. 4) of the queued clusters: argmin over the voxels labelled
// k of (n*x - Sx)^2 + (n*y - Sy)^2 + (n*t - St)^2 in 128-bit integers, ties
// to the smallest voxel index; searched over the window the last assignment
// used and the listed voxels that kept their label for lack of a candidate
// (together they hold S_k), or at set-up over the whole volume.
// ---------------------------------------------------------------------------
struct VBest {
    unsigned long long hi, lo;
    long long p;
};

// Voxel (x, y, t) of index p as a candidate for X_k^* of cluster (n, sx, sy, st).
__device__ __forceinline__ VBest vcandidate(long long p, int x, int y, int t, long long n, long long sx,
                                            long long sy, long long st, bool small)
{
    VBest c;
    c.p = p;
    if (small) {
        const long long dx = n * x - sx, dy = n * y - sy, dt = n * t - st;
        c.hi = 0;
        c.lo = (unsigned long long)(dx * dx) + (unsigned long long)(dy * dy) + (unsigned long long)(dt * dt);
    } else {
        const __int128 dx = (__int128)n * x - sx, dy = (__int128)n * y - sy, dt = (__int128)n * t - st;
        const unsigned __int128 d2 =
            (unsigned __int128)(dx * dx) + (unsigned __int128)(dy * dy) + (unsigned __int128)(dt * dt);
        c.hi = (unsigned long long)(d2 >> 64);
        c.lo = (unsigned long long)d2;
    }
    return c;
}

__device__ __forceinline__ bool vless(const VBest &u, const VBest &v)
{
    return u.hi < v.hi || (u.hi == v.hi && (u.lo < v.lo || (u.lo == v.lo && u.p < v.p)));
}

__device__ __forceinline__ void vshfl_min(VBest &b)
{
    for (int o = 16; o > 0; o >>= 1) {
        VBest c;
        c.hi = __shfl_xor_sync(0xffffffffu, b.hi, o);
        c.lo = __shfl_xor_sync(0xffffffffu, b.lo, o);
        c.p = __shfl_xor_sync(0xffffffffu, b.p, o);
        if (vless(c, b)) b = c;
    }
}

// The `end` voxels of rows of div_w.d and frames of div_h.d rows from (xlo, ylo,
// tlo) for cluster k, thread t of `threads`: eight label loads before any is
// compared, then the matches one by one (compact code: it is cold on every
// launch).
template <bool EXACT>
__device__ __forceinline__ void vproject_scan_rows(const VoxArgs &a, int k, long long n, long long sx, long long sy,
                                                   long long st, bool small, int xlo, int ylo, int tlo, Divisor div_w,
                                                   Divisor div_h, unsigned end, int t, int threads, VBest &b)
{
    constexpr int VB = 8;
    const auto place = [&](unsigned i, int &x, int &y, int &z) {
        int row;
        div_w.split<EXACT>(min(i, end - 1u), row, x);  // (past the end: the last voxel, which changes nothing)
        div_h.split<EXACT>((unsigned)row, z, y);
        x += xlo;
        y += ylo;
        z += tlo;
    };
    for (unsigned base = (unsigned)t; base < end; base += (unsigned)(threads * VB)) {
        unsigned match = 0u;
        int lab[VB], x, y, z;
#pragma unroll
        for (int u = 0; u < VB; ++u) {
            place(base + (unsigned)(u * threads), x, y, z);
            lab[u] = a.labels[((long long)z * a.H + y) * a.W + x];
        }
#pragma unroll
        for (int u = 0; u < VB; ++u) match |= lab[u] == k ? 1u << u : 0u;
        for (; match; match &= match - 1) {
            place(base + (unsigned)((__ffs(match) - 1) * threads), x, y, z);
            const VBest c =
                vcandidate(((long long)z * a.H + y) * a.W + x, x, y, z, n, sx, sy, st, EXACT || small);
            if (vless(c, b)) b = c;
        }
    }
}

// The w x h x d voxels from (xlo, ylo, tlo); the two forms as in 2-D.
__device__ __forceinline__ void vproject_scan(const VoxArgs &a, int k, long long n, long long sx, long long sy,
                                              long long st, bool small, int xlo, int ylo, int tlo, int w, int h,
                                              int d, int t, int threads, VBest &b)
{
    const Divisor div_w((unsigned)max(w, 1)), div_h((unsigned)max(h, 1));
    const unsigned rows = (unsigned)(max(h, 0) * max(d, 0));
    const unsigned end = (unsigned)max(w, 0) * rows;  // (within the volume: at most 2^30)
    if (small && div_w.exact(end) && div_h.exact(rows))
        vproject_scan_rows<true>(a, k, n, sx, sy, st, small, xlo, ylo, tlo, div_w, div_h, end, t, threads, b);
    else
        vproject_scan_rows<false>(a, k, n, sx, sy, st, small, xlo, ylo, tlo, div_w, div_h, end, t, threads, b);
}

// Queue entries j0, j0 + stride, ...: one CTA per queued cluster.  A list of more
// than half the voxels is slower than the volume in order (32 x 240 x 320 with
// 2000 clusters, an iteration with 25, 50 and 90% of the columns in no window:
// 3.19, 4.96 and 5.33 ms; by the list 3.30, 6.51 and 11.31; the volume from
// a quarter on 4.51, 4.99 and 5.34).
constexpr int VPROJ_LIST_SHIFT = 1;

__device__ __forceinline__ void vproject_cta(const VoxArgs &a, int whole, int j0, int stride)
{
    __shared__ VBest s_best[VPROJ_THREADS / 32];
    const int nproj = a.ctr->nproj;
    whole |= a.ctr->proj_orphans > a.N >> VPROJ_LIST_SHIFT;
    const int n_orphans = whole ? 0 : a.ctr->proj_orphans;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int j = j0; j < nproj; j += stride) {
        const int k = a.proj_list[j];
        const long long n = a.st_n[k], sx = a.st_sx[k], sy = a.st_sy[k], st = a.st_st[k];
        int xlo = 0, xhi = a.W - 1, ylo = 0, yhi = a.H - 1, tlo = 0, thi = a.T - 1;
        if (!whole) {
            const int *pw = a.prev_win + 6 * (long long)k;
            xlo = pw[0]; xhi = pw[1]; ylo = pw[2]; yhi = pw[3]; tlo = pw[4]; thi = pw[5];
        }
        // 64-bit squared distances when 3 (n * largest dimension)^2 < 2^62
        const double bound = (double)max(a.W, max(a.H, a.T));
        const bool small = 3.0 * ((double)n * bound) * ((double)n * bound) < 4.0e18;
        VBest b = {~0ull, ~0ull, LLONG_MAX};
        vproject_scan(a, k, n, sx, sy, st, small, xlo, ylo, tlo, xhi - xlo + 1, yhi - ylo + 1, thi - tlo + 1, tid,
                      VPROJ_THREADS, b);
        for (int i = tid; i < n_orphans; i += VPROJ_THREADS) {
            const int p = a.orphan_list[i];
            if (a.labels[p] != k) continue;
            const int t = (int)(p / a.HW), q = (int)(p - t * a.HW), y = q / a.W;
            const VBest c = vcandidate(p, q - y * a.W, y, t, n, sx, sy, st, small);
            if (vless(c, b)) b = c;
        }
        vshfl_min(b);
        if (lane == 0) s_best[warp] = b;
        __syncthreads();
        if (warp == 0) {
            b = lane < VPROJ_THREADS / 32 ? s_best[lane] : VBest{~0ull, ~0ull, LLONG_MAX};
            vshfl_min(b);
            if (lane == 0) {
                if (b.p == LLONG_MAX) {
                    atomicExch(&a.ctr->error, ERR_BAD_LABEL);
                } else {
                    const int t = (int)(b.p / a.HW);
                    const long long q = b.p - (long long)t * a.HW;
                    const int y = (int)(q / a.W), x = (int)(q - (long long)y * a.W);
                    a.st_end[k] = make_int4(x, y, t, 0);
                    a.cdev[k].ex = x;
                    a.cdev[k].ey = y;
                    a.cdev[k].et = t;
                }
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(VPROJ_THREADS) k_vproject(VoxArgs a, int whole)
{
    pdl_wait();
    pdl_release();
    vproject_cta(a, whole, blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------------------
// Candidate lists: exclusive scan of the tile counts, then the (cluster, tile)
// slots, one thread each.  The assignment of a tile zeroes its count and
// cursor once it has read its list, so the lists touch nothing the projection
// reads, and both run in one launch (VLISTS_MAX_TILES bounds the scan in shared
// memory, as in 2-D); volumes of more tiles take a scan and a fill kernel after
// the projection.
// ---------------------------------------------------------------------------
constexpr int VSCAN_THREADS = 1024;
// (n + 1) ints of dynamic shared memory beside at most 1020 bytes of the
// projection's static arrays: 48 KB in all, what a launch gets unasked
constexpr int VLISTS_MAX_TILES = 12032;

__device__ __forceinline__ void vfill_slot(const VoxArgs &a, const int *tile_off, long long i)
{
    const unsigned slots = (unsigned)(a.tpw_x * a.tpw_y * a.tpw_t);
    const long long total = (long long)a.Keff * slots;
    if (i >= total) return;
    const int k = total < (1LL << 32) ? (int)((unsigned)i / slots) : (int)(i / slots);
    int j = (int)(i - (long long)k * slots);
    const VoxCluster &cd = a.cdev[k];
    const int xlo = cd.xlo, xhi = cd.xhi, ylo = cd.ylo, yhi = cd.yhi, tlo = cd.tlo, thi = cd.thi;
    if (xlo > xhi || ylo > yhi || tlo > thi) return;
    const int jx = j % a.tpw_x;
    j /= a.tpw_x;
    const int jy = j % a.tpw_y, jt = j / a.tpw_y;
    const int tx = xlo / VTX + jx, ty = ylo / VTY + jy, tt = tlo / VTT + jt;
    if (tx > xhi / VTX || ty > yhi / VTY || tt > thi / VTT) return;
    const int tile = (tt * a.n_ty + ty) * a.n_tx + tx;
    const int pos = tile_off[tile] + atomicAdd(&a.tile_cursor[tile], 1);
    if (pos < a.tile_cap) a.tile_list[pos] = k;
}

__global__ void __launch_bounds__(VSCAN_THREADS) k_vscan(VoxArgs a)
{
    pdl_wait();
    pdl_release();
    __shared__ int s_warp[32];
    const int n = a.n_tx * a.n_ty * a.n_tt;
    cta_scan(a.tile_count, a.tile_off, n, VSCAN_THREADS, s_warp);  // (ends with a barrier)
    // (tile_off[n] is this thread's own write)
    if (threadIdx.x == 0 && a.tile_off[n] > a.tile_cap) atomicExch(&a.ctr->error, ERR_TILE_LIST_OVERFLOW);
}

__global__ void k_vfill(VoxArgs a)
{
    pdl_wait();
    pdl_release();
    vfill_slot(a, a.tile_off, blockIdx.x * (long long)blockDim.x + threadIdx.x);
}

// The lists by CTAs [0, n_lists), placed first, and the projection by the
// others (none without a queue: set_state).
__global__ void __launch_bounds__(VPROJ_THREADS) k_vproject_lists(VoxArgs a, int whole, int n_lists)
{
    pdl_wait();
    pdl_release();
    extern __shared__ int s_off[];
    __shared__ int s_warp[32];
    const int blk = (int)blockIdx.x;
    if (blk >= n_lists) {
        vproject_cta(a, whole, blk - n_lists, (int)gridDim.x - n_lists);
        return;
    }
    const int n = a.n_tx * a.n_ty * a.n_tt;
    cta_scan(a.tile_count, s_off, n, VPROJ_THREADS, s_warp);
    if (blk == 0) {
        for (int i = threadIdx.x; i <= n; i += VPROJ_THREADS) a.tile_off[i] = s_off[i];
        if (threadIdx.x == 0 && s_off[n] > a.tile_cap) atomicExch(&a.ctr->error, ERR_TILE_LIST_OVERFLOW);
    }
    const long long slots = (long long)a.Keff * a.tpw_x * a.tpw_y * a.tpw_t;
    for (long long i = blk * (long long)VPROJ_THREADS + threadIdx.x; i < slots; i += (long long)n_lists * VPROJ_THREADS)
        vfill_slot(a, s_off, i);
}

// ---------------------------------------------------------------------------
// Assignment: one voxel per thread, every candidate of the tile whose window
// holds it, the smallest (D, k).  The path sums follow the 3-D stepping rule
// in walk order, FP32.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int vpath_sums(const float4 *__restrict__ plane, int W, long long HW, int px,
                                          int py, int pt, int ex, int ey, int et, float cL, float ca,
                                          float cb, float &sum_dc, float &sum_w)
{
    const int dx = ex - px, dy = ey - py, dt = et - pt;
    const int first = dx ? dx : dy ? dy : dt;  // below zero: the endpoint is the smaller end
    const int adx = abs(dx), ady = abs(dy), adt = abs(dt);
    // strides (elements) of the three axes with their signs along the walk (x
    // never falls); the major axis is the first largest |delta|.  A volume
    // holds at most 2^30 voxels, so offsets and strides are 32-bit.
    const int hw = (int)HW;
    const int sxs = 1, sys = (dy ^ first) < 0 ? -W : W, sts = (dt ^ first) < 0 ? -hw : hw;
    int ns, d1, d2, smaj, s1, s2;
    if (adx >= ady && adx >= adt) { ns = adx; smaj = sxs; d1 = ady; s1 = sys; d2 = adt; s2 = sts; }
    else if (ady >= adt) { ns = ady; smaj = sys; d1 = adx; s1 = sxs; d2 = adt; s2 = sts; }
    else { ns = adt; smaj = sts; d1 = adx; s1 = sxs; d2 = ady; s2 = sys; }
    int q = first < 0 ? et * hw + ey * W + ex : pt * hw + py * W + px;
    float dc = 0.f, w = 0.f;
    if (ns <= FIXED_STEP_MAX_NS) {
        // the fixed-point rule in closed form per minor axis: sample i lies at
        // q + i smaj + m1_i s1 + m2_i s2 with m_i the high word of
        // 2^31 + i S; four samples per group from the group's accumulators
        const uint32_t S1 = fixed_step_slope(d1, ns), S2 = fixed_step_slope(d2, ns);
        uint32_t a1 = 0x80000000u, a2 = 0x80000000u;
        const int n = ns + 1;
        const auto at = [&](int k) {
            const int m1 = k == 0 ? 0 : (int)(((unsigned long long)S1 * (unsigned)k + a1) >> 32);
            const int m2 = k == 0 ? 0 : (int)(((unsigned long long)S2 * (unsigned)k + a2) >> 32);
            return q + k * smaj + m1 * s1 + m2 * s2;
        };
        int i = 0;
#pragma unroll 1
        for (; i + 4 <= n; i += 4) {
            float4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = __ldg(plane + at(k));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                dc += colour_dist(v[k], cL, ca, cb);
                w += v[k].w;
            }
            const unsigned long long t1 = (unsigned long long)S1 * 4u + a1, t2 = (unsigned long long)S2 * 4u + a2;
            a1 = (uint32_t)t1;
            a2 = (uint32_t)t2;
            q += 4 * smaj + (int)(t1 >> 32) * s1 + (int)(t2 >> 32) * s2;
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (i + k < n) {
                const float4 v = __ldg(plane + at(k));
                dc += colour_dist(v, cL, ca, cb);
                w += v.w;
            }
        sum_dc = dc;
        sum_w = w;
        return n;
    }
    const int two_ns = 2 * ns, two_d1 = 2 * d1, two_d2 = 2 * d2;
    int e1 = ns, e2 = ns;
#pragma unroll 4
    for (int i = 0; i <= ns; ++i) {
        const float4 v = __ldg(plane + q);
        dc += colour_dist(v, cL, ca, cb);
        w += v.w;
        e1 += two_d1;
        e2 += two_d2;
        int step = smaj;
        if (e1 >= two_ns) { e1 -= two_ns; step += s1; }
        if (e2 >= two_ns) { e2 -= two_ns; step += s2; }
        q += step;
    }
    sum_dc = dc;
    sum_w = w;
    return ns + 1;
}

// Candidate clusters of one tile held in shared memory; a tile with more
// evaluates voxel by voxel over the global list instead.
constexpr int VCAND = 128;
constexpr int VQUEUE = 96;  // pairs a warp's queue holds (pass 2)

__device__ __forceinline__ unsigned long long vpack_best(float D, int slot)
{
    return ((unsigned long long)__float_as_uint(D) << 32) | (unsigned)slot;  // D >= 0
}

// Rank of cluster k among the sorted candidate ids, or -1.
__device__ __forceinline__ int vfind_slot(const int *ids, int cnt, int k)
{
    int lo = 0, hi = cnt;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (ids[mid] < k) lo = mid + 1;
        else hi = mid;
    }
    return lo < cnt && ids[lo] == k ? lo : -1;
}

// The assignment of one tile, a voxel per thread, pruned as in 2-D.  Each warp
// (32 voxels, 16 columns x 2 rows of a frame) works alone after the set-up:
// pass 1 evaluates each voxel's previous label (when it is a candidate of the
// voxel); pass 2 checks the other candidates whose boxes meet the warp's
// voxels against a lower bound of D, queues the pairs it cannot rule out and
// walks them 32 at a time.  The bound is the 2-D one with one axis more
// (scalp_assign_tile.cuh: q = P + K + f . g, its rounding covered by the same
// margin), six multiply-adds on values in registers.  Its first form cut each
// candidate's box into 32-voxel items taken from a shared counter, each lane
// reading its voxel's sample and forming both squared distances, behind six
// block barriers instead of one or two: 226 us a launch on 32 x 240 x 320 with
// 2000 clusters, 200 now (185.7 M against 164.3 M warp instructions; the walks
// are most of what is left).
//
// Per candidate (slot c): the record, and for the bound
//   s_rec = (box, K bits, g_x bits, g_y bits), s_col = (c, g_t)
// with the box as one bit per column (0-15), row (16-23) and frame (24-27) of
// the tile.
//
// THIN: a volume of fewer than sixteen columns, or of one row, fills the lanes
// of that layout poorly (and most warps not at all).  The tile's voxels (a.thin_w
// x a.thin_h x a.thin_d, x fastest) are packed into the first warps' lanes then,
// the CTA has no more warps than it can use, and up to half a tile's voxels the
// warps form groups: every group takes the voxels, group g checks the slots = g
// modulo the number of groups against the first group's pass-1 D's, and they
// meet in the voxels' best D.  Six iterations, packed and in the layout above:
// 300 x 700 x 1 with 40 clusters 427 and 1688 us, x 7 1.61 and 2.02 ms (with 300
// clusters), 300 x 300 x 9 684 and 962 us, x 15 1032 and 1139; 2000 x 1 x 600
// 1.30 and 4.95 ms; a line of 60,000 347-814 and 799-2501 us.  Few frames or a
// few rows fill the layout's warps one by one and stay with it (2 x 400 x 600
// 413 us).
template <bool THIN>
__global__ void __launch_bounds__(VTILE) k_vassign(VoxArgs a)
{
    static_assert(VTX == 16 && VTY == 8 && VTT == 4, "a box is 16 + 8 + 4 bits, a warp 16 x 2 voxels");
    __shared__ VoxCluster cand[VCAND];
    __shared__ int4 s_rec[VCAND];
    __shared__ float4 s_col[VCAND];
    __shared__ int s_sorted[VCAND];   // candidate ids in slot order
    __shared__ int s_ids[VCAND];
    __shared__ uint16_t s_queue[VTILE / 32][VQUEUE];  // slot << 5 | lane
    __shared__ unsigned long long s_best[VTILE];
    const unsigned FULL = 0xffffffffu;
    pdl_wait();
    pdl_release();
    const int tile = blockIdx.x;
    const int tx = tile % a.n_tx, ty = (tile / a.n_tx) % a.n_ty, tt = tile / (a.n_tx * a.n_ty);
    const int x0 = tx * VTX, y0 = ty * VTY, t0 = tt * VTT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int blocks = THIN ? (a.thin_w * a.thin_h * a.thin_d + 31) >> 5 : VTILE / 32;  // of 32 voxels
    const int groups = THIN ? (int)(blockDim.x >> 5) / blocks : 1, group = THIN ? warp / blocks : 0;
    const int base = THIN ? warp % blocks * 32 : warp * 32;  // of the warp's voxels in the tile
    // place in the tile of its voxel v
    const auto place = [&](int v, int &vx, int &vy, int &vt) {
        const int row = THIN ? v / a.thin_w : v / VTX;
        vx = THIN ? v - row * a.thin_w : v % VTX;
        vt = THIN ? row / a.thin_h : row / VTY;
        vy = THIN ? row - vt * a.thin_h : row % VTY;
    };
    int lx, ly, lt;
    place(base + lane, lx, ly, lt);
    const int x = x0 + lx, y = y0 + ly, t = t0 + lt;
    const bool inside = x < a.W && y < a.H && t < a.T && (!THIN || (lt < a.thin_d && group < groups));
    const bool valid = inside && group == 0;  // (the voxel's own thread)
    const int off = a.tile_off[tile];
    const int cnt = (int)max(0LL, min((long long)a.tile_off[tile + 1], a.tile_cap) - off);
    const bool fast = cnt <= VCAND;
    if (tid == 0) {  // this tile's list is read: ready the counts for the next update
        a.tile_count[tile] = 0;
        a.tile_cursor[tile] = 0;
        // the last projection completed before this launch: its queue starts again
        if (tile == 0) a.ctr->nproj = 0;
    }
    const long long p = ((long long)t * a.H + y) * a.W + x;
    unsigned my_samples = 0, my_pairs = 0;
    int lab = -1;
    const int prev = fast && valid ? a.labels[p] : -1;  // overlaps the set-up

    if (fast) {
        const auto write_records = [&](int rank, int id, const VoxCluster &cd) {
            cand[rank] = cd;
            s_sorted[rank] = id;
            const int xa = max(cd.xlo, x0), xb = min(min(cd.xhi, x0 + VTX - 1), a.W - 1);
            const int ya = max(cd.ylo, y0), yb = min(min(cd.yhi, y0 + VTY - 1), a.H - 1);
            const int ta = max(cd.tlo, t0), tb = min(min(cd.thi, t0 + VTT - 1), a.T - 1);
            unsigned box = 0u;
            if (xa <= xb && ya <= yb && ta <= tb)
                box = (0xffffffffu >> (31 - (xb - xa))) << (xa - x0) |
                      (0xffffffffu >> (31 - (yb - ya))) << (ya - y0 + 16) |
                      (0xffffffffu >> (31 - (tb - ta))) << (ta - t0 + 24);
            const float kx = cd.xk - (float)x0, ky = cd.yk - (float)y0, kt = cd.tk - (float)t0;
            const float K = BOUND_SCALE * fmaf(a.lam, fmaf(cd.L, cd.L, fmaf(cd.a, cd.a, cd.b * cd.b)),
                                               a.ms2 * fmaf(kx, kx, fmaf(ky, ky, kt * kt)));
            s_rec[rank] = make_int4((int)box, __float_as_int(K), __float_as_int(-2.0f * a.ms2 * kx),
                                    __float_as_int(-2.0f * a.ms2 * ky));
            s_col[rank] = make_float4(cd.L, cd.a, cd.b, -2.0f * a.ms2 * kt);
        };
        // candidates sorted by cluster index (ranks of distinct ids): by one
        // warp with shuffles when they fit its lanes
        if (cnt <= 32) {
            if (warp == 0) {
                int myid = INT_MAX;
                VoxCluster cd;
                if (lane < cnt) {
                    myid = a.tile_list[off + lane];
                    cd = a.cdev[myid];
                }
                int rank = 0;
                for (int j = 0; j < 32; ++j) rank += __shfl_sync(FULL, myid, j) < myid;
                if (lane < cnt) write_records(rank, myid, cd);
            }
        } else {
            int myid = INT_MAX;
            if (tid < cnt) {
                myid = a.tile_list[off + tid];
                s_ids[tid] = myid;
            }
            __syncthreads();
            if (tid < cnt) {
                int rank = 0;
                for (int j = 0; j < cnt; ++j) rank += s_ids[j] < myid;
                write_records(rank, myid, a.cdev[myid]);
            }
        }
        __syncthreads();
        // D of the warp's voxel v (a lane) for candidate slot c
        const int wy = y0 + (ly & ~1);  // the warp's first row
        const auto evaluate = [&](int v, int c, int &len) {
            const VoxCluster &cd = cand[c];
            int qx = x0 + (v & 15), qy = wy + (v >> 4), qt = t;
            if (THIN) {
                place(base + v, qx, qy, qt);
                qx += x0;
                qy += y0;
                qt += t0;
            }
            const float dcp = colour_dist(__ldg(a.plane + ((long long)qt * a.H + qy) * a.W + qx), cd.L, cd.a, cd.b);
            float sdc, sw;
            len = vpath_sums(a.plane, a.W, a.HW, qx, qy, qt, cd.ex, cd.ey, cd.et, cd.L, cd.a, cd.b, sdc, sw);
            const float ddx = (float)qx - cd.xk, ddy = (float)qy - cd.yk, ddt = (float)qt - cd.tk;
            return scalp_distance(dcp, sdc, sw, len, a.lam, a.gamma, a.ms2, fmaf(ddx, ddx, fmaf(ddy, ddy, ddt * ddt)));
        };
        const auto count_pair = [&](int len) {
            my_samples += len;
            my_pairs += 1;
        };
        // pass 1: the previous label, when the voxel is in its box
        // (a lane without a voxel has no bits, and is in no box)
        const unsigned bits = THIN && !inside ? 0u : 1u << lx | 1u << (16 + ly) | 1u << (24 + lt);
        int slot = prev >= 0 ? vfind_slot(s_sorted, cnt, prev) : -1;
        if (slot >= 0 && ((unsigned)s_rec[slot].x & bits) != bits) slot = -1;
        float dprev = __int_as_float(0x7fffffff);  // NaN: none
        unsigned long long mine = ~0ull;
        if (slot >= 0) {
            int len;
            dprev = evaluate(lane, slot, len);
            mine = vpack_best(dprev, slot);
            count_pair(len);
        }
        if (group == 0) s_best[base + lane] = mine;
        if (THIN) {
            __syncthreads();
            if (group > 0 && inside) {  // (the first group's pass 1; ~0: a NaN, and no slot)
                mine = s_best[base + lane];
                dprev = __uint_as_float((unsigned)(mine >> 32));
                slot = (int)(unsigned)mine;
            }
            __syncthreads();  // the D's before any group lowers them
        } else {
            __syncwarp();
        }
        // pass 2: the other candidates
        uint16_t *wq = s_queue[warp];
        const unsigned warp_rows = 3u << (16 + (ly & ~1)), warp_frame = 1u << (24 + lt);
        const unsigned warp_bits = THIN ? __reduce_or_sync(FULL, bits) : 0u;
        int queued = 0, c0 = -32;  // warp-uniform, as all that follows
        unsigned any = 0u;         // candidates c0 + bit that meet the warp's voxels and are left
        for (bool more = true; more;) {
            const float X = (float)lx, Y = (float)ly, Z = (float)lt;
            float fL, fa, fb, thr;
            {
                const float4 v = inside ? __ldg(a.plane + p) : make_float4(0.f, 0.f, 0.f, 0.f);
                thr = bound_threshold(dprev, fmaf(a.lam, fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z)),
                                                  a.ms2 * fmaf(X, X, fmaf(Y, Y, Z * Z))));
                fL = -2.0f * a.lam * v.x;
                fa = -2.0f * a.lam * v.y;
                fb = -2.0f * a.lam * v.z;
            }
            const unsigned lanes_below = (1u << lane) - 1u;
            while (queued <= VQUEUE - 32) {
                if (!any) {
                    c0 += 32;
                    more = c0 < cnt;
                    if (!more) break;
                    const unsigned m = c0 + lane < cnt ? (unsigned)s_rec[c0 + lane].x : 0u;
                    if (THIN) {
                        const unsigned meet = m & warp_bits;
                        any = __ballot_sync(FULL, (meet & 0xffffu) && (meet & 0xff0000u) && (meet & 0xf000000u) &&
                                                      (c0 + lane) % groups == group);
                    } else {
                        any = __ballot_sync(FULL, (m & warp_rows) && (m & warp_frame));
                    }
                    continue;
                }
                const int c = c0 + __ffs(any) - 1;
                any &= any - 1;
                const int4 r = s_rec[c];
                const float4 ck = s_col[c];
                // (a voxel of the box lies in the volume)
                const bool in = ((unsigned)r.x & bits) == bits && c != slot && (!THIN || bits);
                const float bound =
                    fmaf(fL, ck.x, fmaf(fa, ck.y, fmaf(fb, ck.z, fmaf(X, __int_as_float(r.z),
                                        fmaf(Y, __int_as_float(r.w), fmaf(Z, ck.w, __int_as_float(r.y)))))));
                const bool loses = bound > thr;
                if (a.count_samples && in && loses) {
                    // a pair that cannot win is not walked (counted as the method's work)
                    const VoxCluster &cd = cand[c];
                    count_pair(max(abs(x - cd.ex), max(abs(y - cd.ey), abs(t - cd.et))) + 1);
                }
                const bool keep = in && !loses;
                const unsigned kept = __ballot_sync(FULL, keep);
                if (keep) wq[queued + __popc(kept & lanes_below)] = (uint16_t)(c << 5 | lane);
                queued += __popc(kept);
            }
            __syncwarp();  // the queued pairs
            int done = 0;
#pragma unroll 1
            for (; more ? done + 32 <= queued : done < queued; done += 32) {
                if (done + lane >= queued) continue;
                const int e = wq[done + lane], v = e & 31, c = e >> 5;
                int len;
                const float D = evaluate(v, c, len);
                atomicMin(&s_best[base + v], vpack_best(D, c));
                count_pair(len);
            }
            if (more) {  // the pairs left over start the next queue
                queued -= done;
                const uint16_t e = lane < queued ? wq[done + lane] : (uint16_t)0;
                __syncwarp();
                if (lane < queued) wq[lane] = e;
                __syncwarp();
            }
        }
        if (THIN) __syncthreads();
        else __syncwarp();
        if (valid) {
            const unsigned long long bb = s_best[base + lane];
            // slot -> cluster index (the record's pad field holds k)
            if (bb != ~0ull) lab = cand[(int)(bb & 0xffffffffu)].pad;
        }
    } else {
        const float4 own = valid ? __ldg(a.plane + p) : make_float4(0.f, 0.f, 0.f, 0.f);
        float bestD = FLT_MAX;
        int bestk = INT_MAX;
        for (int i = 0; i < cnt; ++i) {
            const int k = a.tile_list[off + i];
            const VoxCluster cd = a.cdev[k];
            if (!valid || x < cd.xlo || x > cd.xhi || y < cd.ylo || y > cd.yhi || t < cd.tlo || t > cd.thi)
                continue;
            float sdc, sw;
            const int len = vpath_sums(a.plane, a.W, a.HW, x, y, t, cd.ex, cd.ey, cd.et, cd.L, cd.a, cd.b,
                                       sdc, sw);
            const float dcp = colour_dist(own, cd.L, cd.a, cd.b);
            const float ddx = (float)x - cd.xk, ddy = (float)y - cd.yk, ddt = (float)t - cd.tk;
            const float ds = fmaf(ddx, ddx, fmaf(ddy, ddy, ddt * ddt));
            const float D = scalp_distance(dcp, sdc, sw, len, a.lam, a.gamma, a.ms2, ds);
            if (D < bestD || (D == bestD && k < bestk)) {
                bestD = D;
                bestk = k;
            }
            my_samples += len;
            my_pairs += 1;
        }
        if (bestk != INT_MAX) lab = bestk;
    }
    if (valid) {
        if (lab >= 0) {
            a.labels[p] = lab;
        } else {
            lab = a.labels[p];  // no window reaches the voxel: keep its label
            a.orphan_list[atomicAdd(&a.ctr->orphans, 1)] = (int)p;
        }
    }
    // a warp = 32 voxels of one frame: 16 columns x 2 rows (THIN: any of the tile)
    const float4 own = valid ? __ldg(a.plane + p) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (THIN) vaggregate(a, valid, lab, x0, y0, t0, lx, ly, lt, own);
    else vaggregate(a, valid, lab, x0, y0 + (ly & ~1), t, lx, ly & 1, 0, own);
    if (a.count_samples) {
        for (int o = 16; o > 0; o >>= 1) {
            my_samples += __shfl_down_sync(0xffffffffu, my_samples, o);
            my_pairs += __shfl_down_sync(0xffffffffu, my_pairs, o);
        }
        if (lane == 0) {
            atomicAdd(&a.ctr->samples, (unsigned long long)my_samples);
            atomicAdd(&a.ctr->pairs, (unsigned long long)my_pairs);
        }
    }
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
constexpr size_t VALIGN = 256;

size_t vcarve(size_t &cur, size_t bytes)
{
    const size_t at = (cur + VALIGN - 1) & ~(VALIGN - 1);
    cur = at + bytes;
    return at;
}

struct VLayout {
    size_t rgb, contour, plane, labels, st_n, st_sx, st_sy, st_st, st_col, st_end, cdev, acc, prev_win,
        proj, tile_count, tile_off, tile_cursor, tile_list, ctr, total;
    long long tile_cap;
    int n_tx, n_ty, n_tt, tpw_x, tpw_y, tpw_t;
};

// Tiles one window can span along an axis: the window holds at most
// floor(2r) + 1 consecutive voxels (one more allowed for rounding).
int vtiles_per_window(double r, int tile)
{
    const long long len = (long long)(2.0 * r) + 2;
    return (int)((len + tile - 1) / tile + 1);
}

bool vsizes_ok(int T, int H, int W, int K)
{
    if (T < 1 || H < 1 || W < 1 || K < 1) return false;
    const long long N = (long long)T * H * W;
    if (N > (1LL << 30) || W > 65535 || H > 65535 || T > 65535) return false;
    return K <= N;
}

void vgrid(int T, int H, int W, int K, int &nx, int &ny, int &nt, double &r)
{
    const double N = (double)T * (double)H * (double)W;
    r = std::cbrt(N / (double)K);
    const int d[3] = {W, H, T};
    int g[3];
    for (int i = 0; i < 3; ++i) {
        g[i] = (int)std::floor((double)d[i] / r + 0.5);
        g[i] = std::max(1, std::min(g[i], d[i]));
    }
    nx = g[0];
    ny = g[1];
    nt = g[2];
}

VLayout vmake_layout(int T, int H, int W, int K)
{
    VLayout L{};
    const size_t N = (size_t)T * H * W;
    int nx, ny, nt;
    double r;
    vgrid(T, H, W, K, nx, ny, nt, r);
    const size_t Keff = (size_t)nx * ny * nt;
    L.n_tx = (W + VTX - 1) / VTX;
    L.n_ty = (H + VTY - 1) / VTY;
    L.n_tt = (T + VTT - 1) / VTT;
    L.tpw_x = std::min(vtiles_per_window(r, VTX), L.n_tx);
    L.tpw_y = std::min(vtiles_per_window(r, VTY), L.n_ty);
    L.tpw_t = std::min(vtiles_per_window(r, VTT), L.n_tt);
    L.tile_cap = (long long)Keff * L.tpw_x * L.tpw_y * L.tpw_t;
    const size_t n_tiles = (size_t)L.n_tx * L.n_ty * L.n_tt;
    size_t cur = 0;
    L.rgb = vcarve(cur, 3 * N);
    L.contour = vcarve(cur, 4 * N);
    L.plane = vcarve(cur, 16 * N);
    L.labels = vcarve(cur, 4 * N);
    L.st_n = vcarve(cur, 8 * Keff);
    L.st_sx = vcarve(cur, 8 * Keff);
    L.st_sy = vcarve(cur, 8 * Keff);
    L.st_st = vcarve(cur, 8 * Keff);
    L.st_col = vcarve(cur, 16 * Keff);
    L.st_end = vcarve(cur, 16 * Keff);
    L.cdev = vcarve(cur, sizeof(VoxCluster) * Keff);
    L.acc = vcarve(cur, sizeof(VoxAcc) * Keff);
    L.prev_win = vcarve(cur, 24 * Keff);
    L.proj = vcarve(cur, 4 * Keff);
    L.tile_count = vcarve(cur, 4 * n_tiles);
    L.tile_off = vcarve(cur, 4 * (n_tiles + 1));
    L.tile_cursor = vcarve(cur, 4 * n_tiles);
    L.tile_list = vcarve(cur, 4 * (size_t)L.tile_cap);
    L.ctr = vcarve(cur, sizeof(DevCounters));
    L.total = (cur + VALIGN - 1) & ~(VALIGN - 1);
    return L;
}

}  // namespace
}  // namespace scalp

using namespace scalp;

struct scalp_vctx {
    int T, H, W, K;
    long long N;
    int nx, ny, nt, Keff;
    double r, gamma;
    float m;
    cudaStream_t st;
    unsigned char *ws;
    VLayout L;
    VoxArgs a;
    int thin_threads;  // of an assignment CTA that packs its tile (0: a voxel per thread)
    int iterations;
    // profiling: an event pair around each assignment launch
    bool profiling = false;
    std::vector<cudaEvent_t> ev;
    int ev_pending = 0;  // pairs recorded and not yet read
    double prof_ms = 0.0;
    long long prof_launches = 0;
};

namespace {

thread_local std::string g_verr;

int vfail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    g_verr = buf;
    scalp::set_last_error(buf);
    return code;
}

int vcheck(cudaError_t e, const char *what)
{
    return e == cudaSuccess ? SCALP_OK : vfail(SCALP_E_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

// Programmatic launches (each kernel placed while the one before drains),
// except around the profiling event records.
void venqueue_update(scalp_vctx *c, int from_acc, int whole)
{
    const bool pdl = !c->profiling;
    const long long threads = (long long)c->Keff * VUPDATE_LANES;
    pdl_launch(pdl, k_vupdate, dim3((unsigned)ceil_div_ll(threads, VUPDATE_THREADS)), dim3(VUPDATE_THREADS), 0, c->st,
               c->a, from_acc);
    const int n = c->a.n_tx * c->a.n_ty * c->a.n_tt;
    const long long slots = (long long)c->Keff * c->a.tpw_x * c->a.tpw_y * c->a.tpw_t;
    if (n <= VLISTS_MAX_TILES) {
        // one resident wave: list CTAs of four slots per thread, the projection in the rest
        const int n_lists = (int)std::max(std::min(ceil_div_ll(slots, 4LL * VPROJ_THREADS), 64LL), 1LL);
        const int n_proj = from_acc ? std::max(std::min(c->Keff, 2 * 152 - n_lists), 1) : 0;
        pdl_launch(pdl, k_vproject_lists, dim3((unsigned)(n_lists + n_proj)), dim3(VPROJ_THREADS),
                   (size_t)(n + 1) * sizeof(int), c->st, c->a, whole, n_lists);
        return;
    }
    if (from_acc)
        pdl_launch(pdl, k_vproject, dim3(std::min(c->Keff, 2 * 152)), dim3(VPROJ_THREADS), 0, c->st, c->a,
                   whole);
    pdl_launch(pdl, k_vscan, dim3(1), dim3(VSCAN_THREADS), 0, c->st, c->a);
    pdl_launch(pdl, k_vfill, dim3((unsigned)((slots + 255) / 256)), dim3(256), 0, c->st, c->a);
}

// The counters go to the thread's pinned status buffer behind the stream's
// work: one asynchronous copy and one synchronisation.
int vdevice_status(scalp_vctx *c)
{
    DevCounters local;
    DevCounters *h = pinned_status_buffer();
    if (!h) h = &local;
    int rc = vcheck(cudaMemcpyAsync(h, c->a.ctr, sizeof(DevCounters), cudaMemcpyDeviceToHost, c->st),
                    "read counters");
    if (rc) return rc;
    rc = vcheck(cudaStreamSynchronize(c->st), "synchronise");
    if (rc) return rc;
    if (h->error) return vfail(SCALP_E_INTERNAL, "device-side check failed (code %d)", h->error);
    return SCALP_OK;
}

}  // namespace

extern "C" {

size_t scalp_voxel_workspace_bytes(int32_t T, int32_t H, int32_t W, int32_t K, const scalp_params *params)
{
    (void)params;
    if (!vsizes_ok(T, H, W, K)) return 0;
    return vmake_layout(T, H, W, K).total;
}

int scalp_voxel_init(scalp_vctx **out, const scalp_volume *vol, int32_t K, float m,
                     const scalp_params *params)
{
    if (!out) return vfail(SCALP_E_ARG, "out is NULL");
    *out = nullptr;
    if (!vol || !vol->rgb || !params) return vfail(SCALP_E_ARG, "volume, volume->rgb and params are required");
    if (!vsizes_ok(vol->T, vol->H, vol->W, K)) return vfail(SCALP_E_ARG, "invalid volume size or K");
    if (!(m > 0.0f)) return vfail(SCALP_E_ARG, "m must be > 0");
    if (params->storage != SCALP_STORAGE_F32) return vfail(SCALP_E_ARG, "supervoxels take FP32 planes only");
    if (params->prior != SCALP_PRIOR_INPUT) return vfail(SCALP_E_ARG, "supervoxels take the input prior only");
    if (!(params->sigma > 0.0f) || params->lambda < 0.0f || params->lambda > 1.0f)
        return vfail(SCALP_E_ARG, "need sigma > 0 and lambda in [0, 1]");
    const size_t need = scalp_voxel_workspace_bytes(vol->T, vol->H, vol->W, K, params);
    if (!params->workspace || params->workspace_bytes < need)
        return vfail(SCALP_E_NOMEM, "supervoxel workspace of %zu bytes needed", need);
    if (reinterpret_cast<uintptr_t>(params->workspace) % VALIGN)
        return vfail(SCALP_E_ARG, "workspace must be 256-byte aligned");
    scalp_vctx *c = new (std::nothrow) scalp_vctx();
    if (!c) return vfail(SCALP_E_NOMEM, "host allocation failed");
    c->T = vol->T; c->H = vol->H; c->W = vol->W; c->K = K; c->m = m;
    c->N = (long long)vol->T * vol->H * vol->W;
    vgrid(c->T, c->H, c->W, K, c->nx, c->ny, c->nt, c->r);
    c->Keff = c->nx * c->ny * c->nt;
    c->gamma = params->gamma < 0.0f ? 2.0 * c->r : (double)params->gamma;
    c->st = reinterpret_cast<cudaStream_t>(params->stream);
    c->ws = reinterpret_cast<unsigned char *>(params->workspace);
    c->L = vmake_layout(c->T, c->H, c->W, K);
    const VLayout &L = c->L;
    VoxArgs &a = c->a;
    a = VoxArgs{};
    a.T = c->T; a.H = c->H; a.W = c->W; a.K = K; a.Keff = c->Keff;
    a.nx = c->nx; a.ny = c->ny; a.nt = c->nt;
    a.N = c->N; a.HW = (long long)c->H * c->W;
    a.r = c->r;
    a.lam = params->lambda;
    a.gamma = (float)c->gamma;
    a.ms2 = (float)((double)m * (double)m / (c->r * c->r));
    a.n_tx = L.n_tx; a.n_ty = L.n_ty; a.n_tt = L.n_tt;
    a.tpw_x = L.tpw_x; a.tpw_y = L.tpw_y; a.tpw_t = L.tpw_t;
    a.tile_cap = L.tile_cap;
    a.thin_w = std::min(c->W, VTX);
    a.thin_h = std::min(c->H, VTY);
    a.thin_d = std::min(c->T, VTT);
    // a voxel per thread, or two groups of warps up to half a tile; the sorting
    // of a tile's candidates takes a thread each (VCAND)
    const int thin = a.thin_w * a.thin_h * a.thin_d, thin_blocks = (thin + 31) / 32;
    c->thin_threads = a.thin_w == VTX && a.thin_h > 1
                          ? 0
                          : std::max(VCAND, thin_blocks * (thin <= VTILE / 2 ? 64 : 32));
    static_assert(VCAND % 32 == 0, "whole warps");
    a.plane = reinterpret_cast<const float4 *>(c->ws + L.plane);
    a.labels = reinterpret_cast<int *>(c->ws + L.labels);
    a.st_n = reinterpret_cast<long long *>(c->ws + L.st_n);
    a.st_sx = reinterpret_cast<long long *>(c->ws + L.st_sx);
    a.st_sy = reinterpret_cast<long long *>(c->ws + L.st_sy);
    a.st_st = reinterpret_cast<long long *>(c->ws + L.st_st);
    a.st_col = reinterpret_cast<float4 *>(c->ws + L.st_col);
    a.st_end = reinterpret_cast<int4 *>(c->ws + L.st_end);
    a.cdev = reinterpret_cast<VoxCluster *>(c->ws + L.cdev);
    a.acc = reinterpret_cast<VoxAcc *>(c->ws + L.acc);
    a.prev_win = reinterpret_cast<int *>(c->ws + L.prev_win);
    // (the contour's staging area, read by the set-up alone)
    a.orphan_list = reinterpret_cast<int *>(c->ws + L.contour);
    a.proj_list = reinterpret_cast<int *>(c->ws + L.proj);
    a.tile_count = reinterpret_cast<int *>(c->ws + L.tile_count);
    a.tile_off = reinterpret_cast<int *>(c->ws + L.tile_off);
    a.tile_cursor = reinterpret_cast<int *>(c->ws + L.tile_cursor);
    a.tile_list = reinterpret_cast<int *>(c->ws + L.tile_list);
    a.ctr = reinterpret_cast<DevCounters *>(c->ws + L.ctr);
    const uint8_t *rgb = vol->rgb;
    const float *con = vol->contour;
    const size_t N = (size_t)c->N;
    int rc = SCALP_OK;
    if (!vol->on_device) {
        rc = vcheck(cudaMemcpyAsync(c->ws + L.rgb, rgb, 3 * N, cudaMemcpyHostToDevice, c->st), "copy volume");
        rgb = c->ws + L.rgb;
        if (!rc && con) {
            rc = vcheck(cudaMemcpyAsync(c->ws + L.contour, con, 4 * N, cudaMemcpyHostToDevice, c->st),
                        "copy contour");
            con = reinterpret_cast<const float *>(c->ws + L.contour);
        }
    }
    const size_t n_tiles = (size_t)L.n_tx * L.n_ty * L.n_tt;
    if (!rc) rc = vcheck(cudaMemsetAsync(a.acc, 0, sizeof(VoxAcc) * c->Keff, c->st), "memset");
    if (!rc) rc = vcheck(cudaMemsetAsync(a.tile_count, 0, 4 * n_tiles, c->st), "memset");
    if (!rc) rc = vcheck(cudaMemsetAsync(a.tile_cursor, 0, 4 * n_tiles, c->st), "memset");
    if (!rc) rc = vcheck(cudaMemsetAsync(a.cdev, 0, sizeof(VoxCluster) * c->Keff, c->st), "memset");
    if (!rc) rc = vcheck(cudaMemsetAsync(a.ctr, 0, sizeof(DevCounters), c->st), "memset");
    if (!rc) rc = vcheck(srgb_table(&a.lut, c->st), "transfer-function table");
    if (rc) {
        delete c;
        return rc;
    }
    k_vsetup<<<152 * 8, 256, 0, c->st>>>(a, rgb, con, params->sigma, reinterpret_cast<float4 *>(c->ws + L.plane));
    venqueue_update(c, 1, 1);
    rc = vcheck(cudaGetLastError(), "initialisation kernels");
    if (!rc) rc = vcheck(cudaStreamSynchronize(c->st), "initialisation");  // host staging is released
    if (rc) {
        delete c;
        return rc;
    }
    c->iterations = 0;
    *out = c;
    return SCALP_OK;
}

int scalp_voxel_iterate(scalp_vctx *c, int32_t n)
{
    if (!c || n < 0) return vfail(SCALP_E_ARG, "ctx is NULL or n < 0");
    for (int i = 0; i < n; ++i) {
        const unsigned tiles = (unsigned)(c->a.n_tx * c->a.n_ty * c->a.n_tt);
        const bool prof = c->profiling;
        if (prof) {
            while ((int)c->ev.size() < 2 * (c->ev_pending + 1)) {
                cudaEvent_t e;
                const int rc = vcheck(cudaEventCreate(&e), "profiling event");
                if (rc) return rc;
                c->ev.push_back(e);
            }
            cudaEventRecord(c->ev[2 * c->ev_pending], c->st);
        }
        pdl_launch(!prof, c->thin_threads ? k_vassign<true> : k_vassign<false>, dim3(tiles),
                   dim3(c->thin_threads ? c->thin_threads : VTILE), 0, c->st, c->a);
        if (prof) cudaEventRecord(c->ev[2 * c->ev_pending++ + 1], c->st);
        venqueue_update(c, 1, 0);
        ++c->iterations;
    }
    return vcheck(cudaGetLastError(), "iteration kernels");
}

int scalp_voxel_labels(scalp_vctx *c, int32_t *out, int32_t out_on_device)
{
    if (!c || !out) return vfail(SCALP_E_ARG, "ctx or out is NULL");
    int rc = vcheck(cudaMemcpyAsync(out, c->a.labels, 4 * (size_t)c->N,
                                    out_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, c->st),
                    "copy labels");
    return rc ? rc : vdevice_status(c);
}

int scalp_voxel_get_info(const scalp_vctx *c, scalp_voxel_info *info)
{
    if (!c || !info) return vfail(SCALP_E_ARG, "ctx or info is NULL");
    info->T = c->T; info->H = c->H; info->W = c->W; info->K = c->K;
    info->nx = c->nx; info->ny = c->ny; info->nt = c->nt; info->Keff = c->Keff;
    info->r = c->r; info->gamma = c->gamma;
    info->iterations = c->iterations;
    return SCALP_OK;
}

int scalp_voxel_get_state(scalp_vctx *c, const scalp_voxel_state *s)
{
    if (!c || !s || !s->labels || !s->n || !s->sx || !s->sy || !s->st || !s->color || !s->endpoint)
        return vfail(SCALP_E_ARG, "ctx and every state array are required");
    const size_t K = (size_t)c->Keff;
    std::vector<float4> col(K);
    std::vector<int4> end(K);
    int rc = vcheck(cudaStreamSynchronize(c->st), "synchronise");
    if (!rc) rc = vcheck(cudaMemcpy(s->labels, c->a.labels, 4 * (size_t)c->N, cudaMemcpyDeviceToHost), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(s->n, c->a.st_n, 8 * K, cudaMemcpyDeviceToHost), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(s->sx, c->a.st_sx, 8 * K, cudaMemcpyDeviceToHost), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(s->sy, c->a.st_sy, 8 * K, cudaMemcpyDeviceToHost), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(s->st, c->a.st_st, 8 * K, cudaMemcpyDeviceToHost), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(col.data(), c->a.st_col, 16 * K, cudaMemcpyDeviceToHost), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(end.data(), c->a.st_end, 16 * K, cudaMemcpyDeviceToHost), "copy");
    if (rc) return rc;
    for (size_t k = 0; k < K; ++k) {
        s->color[3 * k] = col[k].x;
        s->color[3 * k + 1] = col[k].y;
        s->color[3 * k + 2] = col[k].z;
        s->endpoint[3 * k] = end[k].x;
        s->endpoint[3 * k + 1] = end[k].y;
        s->endpoint[3 * k + 2] = end[k].z;
    }
    return vdevice_status(c);
}

int scalp_voxel_set_state(scalp_vctx *c, const scalp_voxel_state *s)
{
    if (!c || !s || !s->labels || !s->n || !s->sx || !s->sy || !s->st || !s->color || !s->endpoint)
        return vfail(SCALP_E_ARG, "ctx and every state array are required");
    const size_t K = (size_t)c->Keff;
    for (size_t k = 0; k < K; ++k) {
        if (s->n[k] < 1 || s->n[k] > (1LL << 30))
            return vfail(SCALP_E_ARG, "cluster %zu has n outside [1, 2^30]", k);
        const long long n = s->n[k];
        if (s->sx[k] < 0 || s->sx[k] > n * (c->W - 1) || s->sy[k] < 0 || s->sy[k] > n * (c->H - 1) ||
            s->st[k] < 0 || s->st[k] > n * (c->T - 1))
            return vfail(SCALP_E_ARG, "barycenter of cluster %zu is outside the volume", k);
        const int32_t *e = s->endpoint + 3 * k;
        if (e[0] < 0 || e[0] >= c->W || e[1] < 0 || e[1] >= c->H || e[2] < 0 || e[2] >= c->T)
            return vfail(SCALP_E_ARG, "endpoint of cluster %zu is outside the volume", k);
    }
    for (long long p = 0; p < c->N; ++p)
        if (s->labels[p] < 0 || s->labels[p] >= c->Keff) return vfail(SCALP_E_ARG, "label out of range");
    std::vector<float4> col(K);
    std::vector<int4> end(K);
    for (size_t k = 0; k < K; ++k) {
        col[k] = make_float4((float)s->color[3 * k], (float)s->color[3 * k + 1], (float)s->color[3 * k + 2], 0.f);
        end[k] = make_int4(s->endpoint[3 * k], s->endpoint[3 * k + 1], s->endpoint[3 * k + 2], 0);
    }
    const size_t n_tiles = (size_t)c->L.n_tx * c->L.n_ty * c->L.n_tt;
    int rc = vcheck(cudaStreamSynchronize(c->st), "synchronise");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.labels, s->labels, 4 * (size_t)c->N, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.st_n, s->n, 8 * K, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.st_sx, s->sx, 8 * K, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.st_sy, s->sy, 8 * K, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.st_st, s->st, 8 * K, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.st_col, col.data(), 16 * K, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemcpy(c->a.st_end, end.data(), 16 * K, cudaMemcpyHostToDevice), "copy");
    if (!rc) rc = vcheck(cudaMemset(c->a.acc, 0, sizeof(VoxAcc) * K), "memset");
    if (!rc) rc = vcheck(cudaMemset(c->a.tile_count, 0, 4 * n_tiles), "memset");
    if (!rc) rc = vcheck(cudaMemset(c->a.tile_cursor, 0, 4 * n_tiles), "memset");
    if (rc) return rc;
    venqueue_update(c, 0, 0);
    rc = vcheck(cudaGetLastError(), "derive kernels");
    return rc ? rc : vdevice_status(c);
}

int scalp_voxel_count_samples(scalp_vctx *c, int32_t enable, int64_t *samples, int64_t *pairs)
{
    if (!c) return vfail(SCALP_E_ARG, "ctx is NULL");
    int rc = vcheck(cudaStreamSynchronize(c->st), "synchronise");
    DevCounters h;
    if (!rc) rc = vcheck(cudaMemcpy(&h, c->a.ctr, sizeof h, cudaMemcpyDeviceToHost), "read counters");
    if (rc) return rc;
    if (samples) *samples = (int64_t)h.samples;
    if (pairs) *pairs = (int64_t)h.pairs;
    if (enable >= 0) {
        if (enable) {
            unsigned long long z[2] = {0, 0};
            rc = vcheck(cudaMemcpy(&c->a.ctr->samples, z, sizeof z, cudaMemcpyHostToDevice), "reset counters");
            if (rc) return rc;
        }
        c->a.count_samples = enable != 0;
    }
    return SCALP_OK;
}

int scalp_voxel_profile(scalp_vctx *c, int32_t enable, double *ms, int64_t *launches)
{
    if (!c) return vfail(SCALP_E_ARG, "ctx is NULL");
    if (c->ev_pending) {
        const int rc = vcheck(cudaStreamSynchronize(c->st), "synchronise");
        if (rc) return rc;
        for (int i = 0; i < c->ev_pending; ++i) {
            float t = 0.f;
            const int r2 = vcheck(cudaEventElapsedTime(&t, c->ev[2 * i], c->ev[2 * i + 1]), "event time");
            if (r2) return r2;
            c->prof_ms += t;
            c->prof_launches += 1;
        }
        c->ev_pending = 0;
    }
    if (ms) *ms = c->prof_ms;
    if (launches) *launches = c->prof_launches;
    if (enable >= 0) {
        if (enable) {
            c->prof_ms = 0.0;
            c->prof_launches = 0;
        }
        c->profiling = enable != 0;
    }
    return SCALP_OK;
}

void scalp_voxel_destroy(scalp_vctx *c)
{
    if (!c) return;
    cudaStreamSynchronize(c->st);
    for (cudaEvent_t e : c->ev) cudaEventDestroy(e);
    delete c;
}

}  // extern "C"
