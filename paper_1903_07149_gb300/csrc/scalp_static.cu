// scalp_static.cu -- scalp_label_means_static(): per-superpixel means with no
// device allocation at all.
//
// Some callers cannot call cudaMalloc or hand the library a workspace: code
// that runs while another component owns the device memory budget, plugins
// that are given only the input and output buffers, or hosts where allocation
// would synchronise the device at a bad moment.  This entry point serves them.
// Its scratch (the integer sums and the sRGB table) is one file-scope
// __device__ array of fixed size, which every GPU that loads the library
// holds until the process exits.  The caller passes only the inputs and the
// output.
#include <algorithm>
#include <cstddef>
#include <cstdarg>
#include <cstdio>
#include <mutex>

#include "../../include/scalp.h"
#include "scalp_launch.h"

using namespace scalp;

namespace {

constexpr int MAX_DEVICES = 64;

// Scratch: SCALP_STATIC_MAX_LABELS cluster sums, then the 256-entry table.
struct StaticScratch {
    ClusterAcc sums[SCALP_STATIC_MAX_LABELS];
    float lut[256];
};
static_assert(offsetof(StaticScratch, sums) == 0, "the sums start the scratch");
static __device__ __align__(256) StaticScratch g_static_scratch;

std::mutex g_static_mutex;
StaticScratch *g_static_ptr[MAX_DEVICES];  // device address, per device, once known

// Errors are reported through scalp_last_error(NULL).
int static_fail(int code, const char *fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    scalp::set_last_error(buf);
    return code;
}

__global__ void k_static_table(StaticScratch *s)
{
    const int i = threadIdx.x;
    if (i < 256) {
        const double c = i / 255.0;
        s->lut[i] = (float)(c <= 0.04045 ? c / 12.92 : pow((c + 0.055) / 1.055, 2.4));
    }
}

// CIELab of 8-bit sRGB (the set-up kernel's conversion), then integer sums per
// label into the static scratch.  Labels outside [0, n_labels) are skipped.
//
// A CTA takes 64 x SUM_CTA_ROWS pixels, a warp 32 columns x SUM_ROWS rows of
// them, a lane one column: it adds up its run of pixels of one label and hands it to a
// small hash table in shared memory when the label changes (places from the
// tile's corner and the halves of the colour sums, so that 32-bit words hold
// the tile's sums).  Each label of the tile then adds its six sums to global
// memory once; a run that finds no place in the table adds its own.  Sums of
// the labels of every 32-pixel row segment instead (warp reductions and six
// atomics per label and row) took 27.8 us on 1080 x 1920 with 2000 labels, the
// table 22.9 us (both with the inputs in DRAM).  What is left is the latency of
// the row steps and of the table's additions: converting two pixels at a time
// with packed instructions changed nothing (23.1).
constexpr int SUM_ROWS = 8, SUM_THREADS = 256, SUM_SLOTS = 256, SUM_PROBES = 8, SUM_BATCH = 4;
constexpr int SUM_CTA_ROWS = SUM_THREADS / 64 * SUM_ROWS;
static_assert(SUM_ROWS * 108LL * (1LL << COLOR_FRAC_BITS) < (1LL << 31), "a run's colour sums");

__global__ void __launch_bounds__(SUM_THREADS)
    k_static_sums(const uint8_t *__restrict__ rgb, long long rgb_stride,
                  const int *__restrict__ labels, int H, int W, int n_labels, StaticScratch *s)
{
    enum { KEY, N, X, Y, L_HI, L_LO, A_HI, A_LO, B_HI, B_LO, WORDS };
    __shared__ float lin[256];
    __shared__ int slot[WORDS][SUM_SLOTS];
    for (int i = threadIdx.x; i < SUM_SLOTS; i += SUM_THREADS) {
        lin[i] = s->lut[i];
        slot[KEY][i] = -1;
        for (int j = 1; j < WORDS; ++j) slot[j][i] = 0;
    }
    __syncthreads();
    static_assert(SUM_SLOTS == 256 && SUM_THREADS == 256, "one table entry and one slot per thread");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned bands = (unsigned)(W + 63) / 64u;
    const int cx = (int)(blockIdx.x % bands) * 64;
    const long long cy = (long long)(blockIdx.x / bands) * SUM_CTA_ROWS;
    const int x = cx + (warp & 1) * 32 + lane;
    const int y0 = (int)min(cy + (warp >> 1) * SUM_ROWS, (long long)H), y1 = min(H, y0 + SUM_ROWS);
    const float scale = (float)(1 << COLOR_FRAC_BITS);
    int run = -1, n = 0, sy = 0, sL = 0, sa = 0, sb = 0;  // sy: rows from y0
    const auto hand_over = [&]() {
        unsigned h = (unsigned)run * 2654435761u >> 24;
        for (int i = 0; i < SUM_PROBES; ++i, h = (h + 1) % SUM_SLOTS) {
            int was = slot[KEY][h];
            if (was == -1) was = atomicCAS(&slot[KEY][h], -1, run);
            if (was == -1 || was == run) {
                atomicAdd(&slot[N][h], n);
                atomicAdd(&slot[X][h], n * (x - cx));
                atomicAdd(&slot[Y][h], n * (int)(y0 - cy) + sy);
                atomicAdd(&slot[L_HI][h], sL >> 16);
                atomicAdd(&slot[L_LO][h], sL & 0xffff);
                atomicAdd(&slot[A_HI][h], sa >> 16);
                atomicAdd(&slot[A_LO][h], sa & 0xffff);
                atomicAdd(&slot[B_HI][h], sb >> 16);
                atomicAdd(&slot[B_LO][h], sb & 0xffff);
                return;
            }
        }
        acc_add(&s->sums[run], n, (long long)n * x, (long long)n * y0 + sy, sL, sa, sb);
    };
    if (x < W) {
        // SUM_BATCH rows are read before any is used (past the last row: that
        // row again)
        for (int yb = y0; yb < y1; yb += SUM_BATCH) {
            int label[SUM_BATCH];
            uint8_t px[SUM_BATCH][3];
#pragma unroll
            for (int u = 0; u < SUM_BATCH; ++u) {
                const int y = min(yb + u, y1 - 1);
                label[u] = labels[(long long)y * W + x];
                const uint8_t *q = rgb + y * rgb_stride + 3 * (long long)x;
                px[u][0] = q[0];
                px[u][1] = q[1];
                px[u][2] = q[2];
            }
            static_assert(SUM_BATCH % 2 == 0, "rows are converted in pairs");
            float3 c[SUM_BATCH];
#pragma unroll
            for (int u = 0; u < SUM_BATCH; u += 2) srgb_to_lab2(lin, px[u], px[u + 1], c[u], c[u + 1]);
#pragma unroll
            for (int u = 0; u < SUM_BATCH; ++u) {
                if (yb + u >= y1) break;
                const int k = label[u] < n_labels ? label[u] : -1;
                if (k != run) {
                    if (run >= 0) hand_over();
                    run = k;
                    n = sy = sL = sa = sb = 0;
                }
                n += 1;
                sy += yb + u - y0;
                sL += __float2int_rn(c[u].x * scale);
                sa += __float2int_rn(c[u].y * scale);
                sb += __float2int_rn(c[u].z * scale);
            }
        }
        if (run >= 0) hand_over();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SUM_SLOTS; i += SUM_THREADS) {
        const int k = slot[KEY][i];
        if (k < 0) continue;
        const long long c = slot[N][i];
        acc_add(&s->sums[k], c, c * cx + slot[X][i], c * cy + slot[Y][i],
                slot[L_HI][i] * 65536LL + slot[L_LO][i], slot[A_HI][i] * 65536LL + slot[A_LO][i],
                slot[B_HI][i] * 65536LL + slot[B_LO][i]);
    }
}

// out[6k .. 6k+5] = (n, mean L, mean a, mean b, mean x, mean y); zeros if n = 0.
// One thread per value (the FP64 divisions of a label side by side).
__global__ void __launch_bounds__(192) k_static_means(const StaticScratch *s, int n_labels, double *out)
{
    pdl_wait();
    const int i = blockIdx.x * 192 + (int)threadIdx.x;
    const int k = i / 6, j = i - 6 * k;
    if (k >= n_labels) return;
    const ClusterAcc &c = s->sums[k];
    const long long n = (long long)c.n;
    const long long v = (long long)(j == 0 ? c.n : j == 1 ? c.sL : j == 2 ? c.sa : j == 3 ? c.sb : j == 4 ? c.sx : c.sy);
    const double den = j == 0 ? 1.0 : j < 4 ? (double)n * (double)(1 << COLOR_FRAC_BITS) : (double)n;
    out[i] = n == 0 ? 0.0 : (double)v / den;
}

}  // namespace

extern "C" int scalp_label_means_static(const uint8_t *rgb, int64_t rgb_stride, const int32_t *labels,
                                        int32_t H, int32_t W, int32_t n_labels, double *out,
                                        void *stream)
{
    if (!rgb || !labels || !out) return static_fail(SCALP_E_ARG, "rgb, labels and out must be device pointers");
    if (H < 1 || W < 1 || (long long)H * W > (1LL << 30))
        return static_fail(SCALP_E_ARG, "need H, W >= 1 and H*W <= 2^30");
    if (n_labels < 1 || n_labels > SCALP_STATIC_MAX_LABELS)
        return static_fail(SCALP_E_ARG, "n_labels must be in [1, %d] (the fixed scratch holds %d)",
                           SCALP_STATIC_MAX_LABELS, SCALP_STATIC_MAX_LABELS);
    if (rgb_stride != 0 && rgb_stride < 3LL * W) return static_fail(SCALP_E_ARG, "rgb_stride < 3*W");
    const long long stride = rgb_stride ? rgb_stride : 3LL * W;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return static_fail(SCALP_E_CUDA, "cudaGetDevice: %s", cudaGetErrorString(e));
    if (dev < 0 || dev >= MAX_DEVICES) return static_fail(SCALP_E_ARG, "device %d not supported", dev);
    StaticScratch *s;
    {
        // set-up, once per device, with that device current: the scratch's
        // device address (the symbol itself is only a host-side stand-in)
        // and the sRGB table
        std::lock_guard<std::mutex> lock(g_static_mutex);
        if (!g_static_ptr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_static_scratch);
            if (e != cudaSuccess)
                return static_fail(SCALP_E_CUDA, "cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            k_static_table<<<1, 256, 0, st>>>(static_cast<StaticScratch *>(p));
            e = cudaGetLastError();
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // ready for any stream
            if (e != cudaSuccess) return static_fail(SCALP_E_CUDA, "table kernel: %s", cudaGetErrorString(e));
            g_static_ptr[dev] = static_cast<StaticScratch *>(p);
        }
        s = g_static_ptr[dev];
    }
    // the sums start at zero on every call
    e = cudaMemsetAsync(static_cast<void *>(s), 0, sizeof(ClusterAcc) * (size_t)n_labels, st);
    if (e != cudaSuccess) return static_fail(SCALP_E_CUDA, "clear scratch: %s", cudaGetErrorString(e));
    const long long blocks = (long long)((W + 63) / 64) * ((H + SUM_CTA_ROWS - 1) / SUM_CTA_ROWS);
    k_static_sums<<<(unsigned)blocks, SUM_THREADS, 0, st>>>(rgb, stride, labels, H, W, n_labels, s);
    pdl_launch(true, k_static_means, dim3((unsigned)(n_labels + 31) / 32), dim3(192), 0, st,
               (const StaticScratch *)s, n_labels, out);
    e = cudaGetLastError();
    if (e != cudaSuccess) return static_fail(SCALP_E_CUDA, "means kernels: %s", cudaGetErrorString(e));
    return SCALP_OK;
}
