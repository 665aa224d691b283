// scalp_metrics.cu -- maps and scores computed from decompositions.
//
// scalp_quality_metrics: the superpixel metrics of Sec. III-A2 against a
// ground-truth segmentation: boundary recall (Eq. 5), achievable segmentation
// accuracy (Eq. 6), undersegmentation error (Eq. 7) and compactness (Eq. 8).
//
// scalp_boundary_map: the multi-scale boundary confidence map the paper's
// precision-recall evaluation uses (Sec. III-A2: boundary maps of the
// decompositions at several scales, averaged).  A pixel is a boundary pixel of
// a decomposition iff one of its 4-neighbours carries another label; the map
// is the fraction of the decompositions in which it is one.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdarg>
#include <cstdio>

#include "../../include/scalp.h"
#include "scalp_launch.h"

using namespace scalp;

namespace {

struct MapPtrs {
    const int *p[SCALP_MAX_MAPS];
};

__global__ void k_boundary_map(MapPtrs m, int count, int H, int W, float *__restrict__ out)
{
    const long long N = (long long)H * W;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N;
         p += (long long)gridDim.x * blockDim.x) {
        const int y = (int)((unsigned)p / (unsigned)W), x = (int)p - y * W;  // N <= 2^30
        int hits = 0;
        for (int i = 0; i < count; ++i) {
            const int *__restrict__ l = m.p[i];
            const int c = l[p];
            const bool b = (x > 0 && l[p - 1] != c) || (x < W - 1 && l[p + 1] != c) ||
                           (y > 0 && l[p - W] != c) || (y < H - 1 && l[p + W] != c);
            hits += b;
        }
        out[p] = (float)hits / (float)count;
    }
}

int metrics_fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    scalp::set_last_error(buf);
    return code;
}

}  // namespace

extern "C" int scalp_boundary_map(const int32_t *const *labels, int32_t count, int32_t H, int32_t W,
                                  float *out, void *stream)
{
    if (!labels || !out) return metrics_fail(SCALP_E_ARG, "labels and out are required");
    if (count < 1 || count > SCALP_MAX_MAPS)
        return metrics_fail(SCALP_E_ARG, "count must be in [1, %d]", SCALP_MAX_MAPS);
    if (H < 1 || W < 1 || (long long)H * W > (1LL << 30)) return metrics_fail(SCALP_E_ARG, "bad H, W");
    MapPtrs m{};
    for (int i = 0; i < count; ++i) {
        if (!labels[i]) return metrics_fail(SCALP_E_ARG, "labels[%d] is NULL", i);
        m.p[i] = labels[i];
    }
    const long long N = (long long)H * W;
    const int blocks = (int)std::min<long long>((N + 255) / 256, 152 * 16);
    k_boundary_map<<<blocks, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(m, count, H, W, out);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return metrics_fail(SCALP_E_CUDA, "boundary map: %s", cudaGetErrorString(e));
    return SCALP_OK;
}

// ---------------------------------------------------------------------------
// Quality metrics, Eq. 5-8.  Boundary pixels: a 4-neighbour carries another
// label.  BR: ground-truth boundary pixels with a superpixel boundary pixel at
// Euclidean distance < eps.  ASA: sum over superpixels of the largest overlap
// with one segment, over N.  UE: sum over segments and the superpixels that
// meet them of |S_k - G_i|, over N.  CO: (1/N) sum 4 pi |S_k|^2 / |P(S_k)|^2,
// |P| = pixel edges between S_k and the rest (image border included).
// ---------------------------------------------------------------------------
namespace {

struct QualityWs {
    int *ov;                       // n_labels x n_gt overlaps
    unsigned long long *perim;
    long long *best, *ue;          // per superpixel
    double *co;                    // per superpixel
    unsigned long long *counts;    // [0] gt boundary pixels, [1] hits
    double *result;                // br, asa, ue, co
};

// The offsets at distance < eps, as half-widths: row offset dy takes the
// columns within half[|dy|] (-1: none).  Up to QUALITY_RADIUS rows; for larger
// radii k_quality_far tests the distance itself.
constexpr int QUALITY_RADIUS = 15;
struct Disk {
    int r;
    signed char half[QUALITY_RADIUS + 1];
};

// The pixels of both maps in one pass.  A CTA takes 64 x 64 pixels, a warp 32
// columns x QUALITY_ROWS rows of them, a lane one column.
//   * Boundary pixels of the superpixels as one 64-bit mask per row, the
//     warp's columns and 16 on either side, dilated by the disk with shifts;
//     a ground-truth boundary pixel is found iff its bit is set.
//   * Overlaps and perimeters: a lane adds up its run of pixels of one
//     (superpixel, segment) pair and hands it over when the pair changes;
//     the runs that reach the strip's end are merged across the warp first.
//     They are summed in a small hash table in shared memory (a CTA meets
//     some twenty pairs; one that finds no place goes straight to global
//     memory) and added to the global sums once per pair.
// 1080 x 1920, 2000 superpixels with ragged borders: 438 us with one atomic
// per pixel and counter (most of it on the two counters that every pixel
// shares), 27.8 us now: 16.6 MB from DRAM, the rest is the row steps' chain of
// shuffles and ballots.
constexpr int QUALITY_ROWS = 16, QUALITY_THREADS = 256, QUALITY_SLOTS = 256, QUALITY_PROBES = 8;

__global__ void __launch_bounds__(QUALITY_THREADS)
    k_quality_pixels(const int *__restrict__ lab, const int *__restrict__ gt, int n_gt, int H, int W, Disk disk,
                     QualityWs w)
{
    constexpr int WARPS = QUALITY_THREADS / 32;
    __shared__ unsigned long long s_mask[WARPS][QUALITY_ROWS + 2 * QUALITY_RADIUS];
    __shared__ unsigned s_gt[WARPS][QUALITY_ROWS];
    __shared__ unsigned s_count[2];
    __shared__ int s_key[QUALITY_SLOTS], s_n[QUALITY_SLOTS], s_e[QUALITY_SLOTS];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 2) s_count[threadIdx.x] = 0u;
    for (int i = threadIdx.x; i < QUALITY_SLOTS; i += QUALITY_THREADS) {
        s_key[i] = -1;
        s_n[i] = s_e[i] = 0;
    }
    __syncthreads();
    static_assert(WARPS == 8 && QUALITY_ROWS == 16, "a CTA's warps cover 64 x 64 pixels");
    const unsigned bands = (unsigned)(W + 63) / 64u;
    const int x0 = (int)(blockIdx.x % bands) * 64 + (warp & 1) * 32;
    const int y0 = (int)min((long long)(blockIdx.x / bands) * 64 + (warp >> 1) * QUALITY_ROWS, (long long)H);
    const int y1 = min(H, y0 + QUALITY_ROWS);
    const int x = x0 + lane;
    unsigned n_bnd = 0, n_hit = 0;
    int run_key = -1, run_k = 0, run_n = 0, run_e = 0;  // the lane's run: pair, superpixel, pixels, edges
    const auto hand_over = [&](int key, int k, int n, int e) {
        unsigned h = (unsigned)key * 2654435761u >> 24;
        static_assert(QUALITY_SLOTS == 256, "the hash's top eight bits");
        for (int i = 0; i < QUALITY_PROBES; ++i, h = (h + 1) % QUALITY_SLOTS) {
            int was = s_key[h];
            if (was == -1) was = atomicCAS(&s_key[h], -1, key);
            if (was == -1 || was == key) {
                atomicAdd(&s_n[h], n);
                if (e) atomicAdd(&s_e[h], e);
                return;
            }
        }
        atomicAdd(&w.ov[key], n);
        if (e) atomicAdd(&w.perim[k], (unsigned long long)e);
    };
    if (y0 < y1 && x0 < W) {
        // Rows y0 - r .. y1 - 1 + r from top to bottom, each read once: the
        // lane's column of both maps, a column of the 16 on either side of
        // the warp's (superpixels) and of the two next to it (segments).
        // Places outside the image move to its edge, where a neighbour then
        // equals the pixel itself.
        const int r = disk.r, rows = y1 - y0 + 2 * r;
        const bool valid = x < W, halo_valid = lane < 16 ? x >= 16 : x + 16 < W;
        const int xc = min(x, W - 1), xh = lane < 16 ? max(x - 16, 0) : min(x + 16, W - 1);
        const int xg = lane == 0 ? max(x - 1, 0) : lane == 31 ? min(x + 1, W - 1) : xc;
        struct Row {
            int c, h, g, e;  // superpixel: own column, halo column; segment: own column, next to the warp's
        };
        const auto load = [&](int i) {
            const long long o = (long long)min(max(y0 - r + i, 0), H - 1) * W;
            return Row{lab[o + xc], lab[o + xh], gt[o + xc], gt[o + xg]};
        };
        const auto process = [&](int i, const Row &up, const Row &at, const Row &down) {
            const int y = y0 - r + i;
            const bool in = y >= 0 && y < H;
            int l = __shfl_up_sync(FULL, at.c, 1), rt = __shfl_down_sync(FULL, at.c, 1);
            const int h_lo = __shfl_sync(FULL, at.h, 15), h_hi = __shfl_sync(FULL, at.h, 16);
            if (lane == 0) l = h_lo;
            if (lane == 31) rt = h_hi;
            const int e4 = (l != at.c) + (rt != at.c) + (up.c != at.c) + (down.c != at.c);
            int hl = __shfl_up_sync(FULL, at.h, 1), hr = __shfl_down_sync(FULL, at.h, 1);
            const int c_lo = __shfl_sync(FULL, at.c, 0), c_hi = __shfl_sync(FULL, at.c, 31);
            if (lane == 16) hl = c_hi;
            if (lane == 15) hr = c_lo;
            // (bits 0 and 63 lack a neighbour; no disk reaches them)
            const unsigned mc = __ballot_sync(FULL, in && valid && e4);
            const unsigned mh = __ballot_sync(FULL, in && halo_valid && (hl != at.h || hr != at.h || up.h != at.h ||
                                                                         down.h != at.h));
            if (lane == 0)
                s_mask[warp][i] = (mh & 0xffffu) | (unsigned long long)mc << 16 | (unsigned long long)(mh >> 16) << 48;
            if (i < r || i >= rows - r) return;
            int gl = __shfl_up_sync(FULL, at.g, 1), gr = __shfl_down_sync(FULL, at.g, 1);
            if (lane == 0) gl = at.e;
            if (lane == 31) gr = at.e;
            const bool bnd_gt = valid && (gl != at.g || gr != at.g || up.g != at.g || down.g != at.g);
            const unsigned G = __ballot_sync(FULL, bnd_gt);
            if (lane == 0) s_gt[warp][i - r] = G;
            const int e = e4 + (x == 0) + (x == W - 1) + (y == 0) + (y == H - 1);
            const int key = valid ? at.c * n_gt + at.g : -1;  // (n_labels * n_gt <= 2^28)
            if (key != run_key) {
                if (run_key >= 0) hand_over(run_key, run_k, run_n, run_e);
                run_key = key;
                run_k = at.c;
                run_n = run_e = 0;
            }
            run_n += 1;
            run_e += e;
        };
        // four rows at a time, the next four on their way meanwhile
        constexpr int B = 4;
        Row now[B + 2];
#pragma unroll
        for (int u = 0; u < B + 2; ++u) now[u] = load(u - 1);
#pragma unroll 1
        for (int i = 0; i < rows; i += B) {
            Row next[B];
#pragma unroll
            for (int u = 0; u < B; ++u) next[u] = load(i + B + 1 + u);
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (i + u < rows) process(i + u, now[u], now[u + 1], now[u + 2]);
            now[0] = now[B];
            now[1] = now[B + 1];
#pragma unroll
            for (int u = 0; u < B; ++u) now[u + 2] = next[u];
        }
        __syncwarp();
        if (lane < y1 - y0) {
            // row y0 + lane: the dilated boundary against the segments'
            unsigned long long d = 0;
            for (int dy = -r; dy <= r; ++dy) {
                const int h = disk.half[abs(dy)];
                if (h < 0) continue;
                const unsigned long long m = s_mask[warp][lane + r + dy];
                d |= m;
                for (int t = 1; t <= h; ++t) d |= m << t | m >> t;
            }
            const unsigned G = s_gt[warp][lane];
            n_bnd = __popc(G);
            n_hit = __popc(G & (unsigned)(d >> 16));
        }
        __syncwarp();
    }
    // what is left, one hand-over per pair of the warp
    for (unsigned pending = __ballot_sync(FULL, run_key >= 0); pending;) {
        const int leader = __ffs(pending) - 1, key = __shfl_sync(FULL, run_key, leader);
        const unsigned grp = __ballot_sync(FULL, run_key == key);
        const int n = __reduce_add_sync(FULL, run_key == key ? run_n : 0);
        const int e = __reduce_add_sync(FULL, run_key == key ? run_e : 0);
        if (lane == leader) hand_over(key, run_k, n, e);
        pending &= ~grp;
    }
    n_bnd = __reduce_add_sync(FULL, n_bnd);
    n_hit = __reduce_add_sync(FULL, n_hit);
    if (lane == 0 && n_bnd) {
        atomicAdd(&s_count[0], n_bnd);
        atomicAdd(&s_count[1], n_hit);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < QUALITY_SLOTS; i += QUALITY_THREADS) {
        const int key = s_key[i];
        if (key < 0) continue;
        atomicAdd(&w.ov[key], s_n[i]);
        if (s_e[i]) atomicAdd(&w.perim[key / n_gt], (unsigned long long)s_e[i]);
    }
    if (threadIdx.x < 2 && s_count[threadIdx.x])
        atomicAdd(&w.counts[threadIdx.x], (unsigned long long)s_count[threadIdx.x]);
}

// Radii above QUALITY_RADIUS: the ground-truth boundary pixels found, a pixel per
// thread, each searching its own disk row by row until it meets a boundary.
// Bound by the search's loads.  (The warps of k_quality_pixels took their rows
// one after the other, a search a lane, with a square root per offset: a call on
// 1080 x 1920 at eps = 20 3.43 ms against 0.24; 321 x 481 with 4 superpixels at
// eps = 40 63.5 against 1.43, and 9.4 a pixel per thread with the square roots.)
__global__ void __launch_bounds__(256)
    k_quality_far(const int *__restrict__ lab, const int *__restrict__ gt, int H, int W, int r, long long d2_max,
                  QualityWs w)
{
    const long long N = (long long)H * W;
    const auto boundary = [&](const int *__restrict__ l, int x, int y) {
        const long long p = (long long)y * W + x;
        const int c = l[p];
        return (x > 0 && l[p - 1] != c) || (x < W - 1 && l[p + 1] != c) || (y > 0 && l[p - W] != c) ||
               (y < H - 1 && l[p + W] != c);
    };
    unsigned hits = 0;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < N; p += (long long)gridDim.x * blockDim.x) {
        const int y = (int)((unsigned)p / (unsigned)W), x = (int)p - y * W;  // N <= 2^30
        if (!boundary(gt, x, y)) continue;
        bool found = false;
        for (int dy = max(-r, -y); dy <= min(r, H - 1 - y) && !found; ++dy) {
            const long long left = d2_max - (long long)dy * dy;
            if (left < 0) continue;
            long long h = (long long)sqrt((double)left);  // (the disk's half-width here, exactly)
            while (h * h > left) --h;
            while ((h + 1) * (h + 1) <= left) ++h;
            const int last = (int)min(h, (long long)(W - 1 - x));
            for (int dx = -(int)min(h, (long long)x); dx <= last && !found; ++dx) found = boundary(lab, x + dx, y + dy);
        }
        hits += found;
    }
    hits = __reduce_add_sync(0xffffffffu, hits);
    if ((threadIdx.x & 31) == 0 && hits) atomicAdd(&w.counts[1], (unsigned long long)hits);
}

// One warp per superpixel: its row of overlaps gives its size (their sum), the
// largest, and the sum of |S_k| - o over the o > 0.
__global__ void __launch_bounds__(256) k_quality_rows(int n_labels, int n_gt, QualityWs w)
{
    pdl_wait();
    const int k = blockIdx.x * (int)(blockDim.x / 32) + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k >= n_labels) return;
    unsigned a = 0, best = 0, met = 0;
    for (int i = lane; i < n_gt; i += 32) {
        const unsigned o = (unsigned)w.ov[(long long)k * n_gt + i];
        a += o;
        best = max(best, o);
        met += o > 0;
    }
    a = __reduce_add_sync(0xffffffffu, a);
    best = __reduce_max_sync(0xffffffffu, best);
    met = __reduce_add_sync(0xffffffffu, met);
    if (lane == 0) {
        w.best[k] = best;
        w.ue[k] = (long long)a * met - a;
        const double pr = (double)w.perim[k], area = (double)a;
        w.co[k] = a > 0 ? 4.0 * M_PI * area * area / (pr * pr) : 0.0;
    }
}

// One CTA, a fixed summation order: deterministic.
__global__ void __launch_bounds__(1024) k_quality_total(int n_labels, long long N, QualityWs w)
{
    pdl_wait();
    __shared__ long long s_best[1024], s_ue[1024];
    __shared__ double s_co[1024];
    long long b = 0, u = 0;
    double c = 0.0;
    for (int k = threadIdx.x; k < n_labels; k += 1024) {
        b += w.best[k];
        u += w.ue[k];
        c += w.co[k];
    }
    s_best[threadIdx.x] = b;
    s_ue[threadIdx.x] = u;
    s_co[threadIdx.x] = c;
    __syncthreads();
    for (int h = 512; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            s_best[threadIdx.x] += s_best[threadIdx.x + h];
            s_ue[threadIdx.x] += s_ue[threadIdx.x + h];
            s_co[threadIdx.x] += s_co[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const unsigned long long gb = w.counts[0], hit = w.counts[1];
        w.result[0] = gb ? (double)hit / (double)gb : 1.0;
        w.result[1] = (double)s_best[0] / (double)N;
        w.result[2] = (double)s_ue[0] / (double)N;
        w.result[3] = s_co[0] / (double)N;
    }
}

size_t quality_layout(int n_labels, int n_gt, QualityWs *w, unsigned char *base)
{
    size_t cur = 0;
    auto take = [&](size_t bytes) {
        const size_t off = (cur + 255) & ~(size_t)255;
        cur = off + bytes;
        return base ? base + off : nullptr;
    };
    unsigned char *ov = take((size_t)n_labels * n_gt * sizeof(int));
    unsigned char *perim = take((size_t)n_labels * 8);
    unsigned char *best = take((size_t)n_labels * 8);
    unsigned char *ue = take((size_t)n_labels * 8);
    unsigned char *co = take((size_t)n_labels * 8);
    unsigned char *counts = take(2 * 8);
    unsigned char *result = take(4 * 8);
    if (w) {
        w->ov = reinterpret_cast<int *>(ov);
        w->perim = reinterpret_cast<unsigned long long *>(perim);
        w->best = reinterpret_cast<long long *>(best);
        w->ue = reinterpret_cast<long long *>(ue);
        w->co = reinterpret_cast<double *>(co);
        w->counts = reinterpret_cast<unsigned long long *>(counts);
        w->result = reinterpret_cast<double *>(result);
    }
    return (cur + 255) & ~(size_t)255;
}

}  // namespace

namespace {

// The largest value of two maps of n pixels, raised into best[0] and best[1].
__global__ void __launch_bounds__(512) k_map_maxima(const int *__restrict__ m0, const int *__restrict__ m1, long long n,
                                                    int *best)
{
    __shared__ int s_best[2];
    if (threadIdx.x < 2) s_best[threadIdx.x] = INT_MIN;
    __syncthreads();
    int b0 = INT_MIN, b1 = INT_MIN;
    const bool vec = ((reinterpret_cast<uintptr_t>(m0) | reinterpret_cast<uintptr_t>(m1)) & 15) == 0;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    const long long quads = vec ? n / 4 : 0;
    for (long long i = t; i < quads; i += step) {
        const int4 a = reinterpret_cast<const int4 *>(m0)[i], c = reinterpret_cast<const int4 *>(m1)[i];
        b0 = max(b0, max(max(a.x, a.y), max(a.z, a.w)));
        b1 = max(b1, max(max(c.x, c.y), max(c.z, c.w)));
    }
    for (long long i = 4 * quads + t; i < n; i += step) {
        b0 = max(b0, m0[i]);
        b1 = max(b1, m1[i]);
    }
    b0 = __reduce_max_sync(0xffffffffu, b0);
    b1 = __reduce_max_sync(0xffffffffu, b1);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&s_best[0], b0);
        atomicMax(&s_best[1], b1);
    }
    __syncthreads();
    if (threadIdx.x < 2) atomicMax(&best[threadIdx.x], s_best[threadIdx.x]);
}

}  // namespace

// The label counts of a decomposition and a ground truth, one pass over both
// and one read-back (two library reductions and a stack before).
extern "C" int scalp_label_counts(const int32_t *labels, const int32_t *gt, int64_t pixels, int32_t counts[2],
                                  void *workspace, size_t workspace_bytes, void *stream)
{
    if (!labels || !gt || !counts) return metrics_fail(SCALP_E_ARG, "labels, gt and counts are required");
    if (pixels < 1) return metrics_fail(SCALP_E_ARG, "need at least one pixel");
    if (!workspace || workspace_bytes < 8 || reinterpret_cast<uintptr_t>(workspace) % 4)
        return metrics_fail(SCALP_E_NOMEM, "8 bytes of device workspace needed");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int *best = static_cast<int *>(workspace);
    cudaError_t e = cudaMemsetAsync(best, 0x80, 8, st);  // below every label
    if (e == cudaSuccess) {
        const long long blocks = std::min<long long>((pixels + 4 * 512 - 1) / (4 * 512), 152 * 4);
        k_map_maxima<<<(unsigned)blocks, 512, 0, st>>>(labels, gt, pixels, best);
        e = cudaGetLastError();
    }
    int local[2];
    int *h = reinterpret_cast<int *>(scalp::pinned_status_buffer());
    if (!h) h = local;
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, best, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return metrics_fail(SCALP_E_CUDA, "label counts: %s", cudaGetErrorString(e));
    counts[0] = h[0] + 1;
    counts[1] = h[1] + 1;
    return SCALP_OK;
}

extern "C" size_t scalp_quality_workspace_bytes(int32_t H, int32_t W, int32_t n_labels, int32_t n_gt)
{
    if (H < 1 || W < 1 || n_labels < 1 || n_gt < 1) return 0;
    if ((long long)n_labels * n_gt > (1LL << 28)) return 0;
    return quality_layout(n_labels, n_gt, nullptr, nullptr);
}

extern "C" int scalp_quality_metrics(const int32_t *labels, int32_t n_labels, const int32_t *gt,
                                     int32_t n_gt, int32_t H, int32_t W, double eps, void *workspace,
                                     size_t workspace_bytes, scalp_quality *out, void *stream)
{
    if (!labels || !gt || !out) return metrics_fail(SCALP_E_ARG, "labels, gt and out are required");
    if (!(eps > 0)) return metrics_fail(SCALP_E_ARG, "eps must be > 0");
    const size_t need = scalp_quality_workspace_bytes(H, W, n_labels, n_gt);
    if (need == 0) return metrics_fail(SCALP_E_ARG, "bad sizes (n_labels * n_gt <= 2^28)");
    if (!workspace || workspace_bytes < need)
        return metrics_fail(SCALP_E_NOMEM, "workspace of %zu bytes needed", need);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    QualityWs w;
    quality_layout(n_labels, n_gt, &w, reinterpret_cast<unsigned char *>(workspace));
    cudaError_t e = cudaMemsetAsync(workspace, 0, need, st);
    const long long N = (long long)H * W;
    if (e == cudaSuccess) {
        const int r = (int)std::min(std::ceil(eps), (double)std::max(H, W));
        const bool far = r > QUALITY_RADIUS;
        Disk disk{};
        disk.r = far ? 0 : r;  // (far: no offset, so that no pixel is found)
        for (int dy = 0; dy <= QUALITY_RADIUS; ++dy) {
            disk.half[dy] = -1;
            for (int dx = 0; !far && dx <= r && !(std::sqrt((double)(dx * dx + dy * dy)) >= eps); ++dx)
                disk.half[dy] = (signed char)dx;
        }
        const unsigned blocks = (unsigned)((long long)((W + 63) / 64) * ((H + 63) / 64));
        k_quality_pixels<<<blocks, QUALITY_THREADS, 0, st>>>(labels, gt, n_gt, H, W, disk, w);
        // the largest squared distance below eps (square roots are monotone)
        long long d2_max = 2LL * r * r;
        if (far && !(std::sqrt((double)d2_max) < eps)) {
            long long lo = 0;  // (0 < eps)
            for (long long hi = d2_max; hi - lo > 1;) {
                const long long mid = lo + (hi - lo) / 2;
                if (std::sqrt((double)mid) < eps) lo = mid;
                else hi = mid;
            }
            d2_max = lo;
        }
        if (far)
            k_quality_far<<<(unsigned)std::min<long long>((N + 255) / 256, 152 * 16), 256, 0, st>>>(labels, gt, H, W, r,
                                                                                                    d2_max, w);
        pdl_launch(true, k_quality_rows, dim3((unsigned)((n_labels + 7) / 8)), dim3(256), 0, st, n_labels, n_gt, w);
        pdl_launch(true, k_quality_total, dim3(1), dim3(1024), 0, st, n_labels, N, w);
        e = cudaGetLastError();
    }
    double local[4];
    static_assert(sizeof(DevCounters) >= sizeof local, "the pinned buffer holds the four metrics");
    double *r = reinterpret_cast<double *>(scalp::pinned_status_buffer());
    if (!r) r = local;
    if (e == cudaSuccess) e = cudaMemcpyAsync(r, w.result, sizeof local, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return metrics_fail(SCALP_E_CUDA, "quality metrics: %s", cudaGetErrorString(e));
    out->br = r[0];
    out->asa = r[1];
    out->ue = r[2];
    out->co = r[3];
    return SCALP_OK;
}
