// scalp_assign.cu -- the assignment step of SCALP (Algorithm 1, inner loops)
// restated per tile of pixels, plus the fused partial sums of the update.
//
// Algorithm 1 loops over clusters and, for each pixel of a cluster's
// (2r+1)x(2r+1) window, keeps the cluster with the smallest D(p, C_k) (Eq. 3)
// under a strict '<' in ascending k.  Here each pixel evaluates the same set of
// clusters (those whose window holds it, from its tile's candidate list) and
// keeps the smallest (D, k) pair: the same result, in any evaluation order.
//
// One CTA of 512 threads (two per SM) labels a 32 x 32 tile:
//   1. The tile's candidate clusters are copied to shared memory, sorted by
//      cluster index.
//   2. Distance maps.  For a candidate k, every path from a tile pixel in its
//      window to its endpoint e_k lies in the bounding box of those pixels and
//      e_k.  Over that box the CTA computes once the colour distance
//      d_c(q, C_k) of Eq. 1 and the contour factor w(q) of Eq. 2 (an FP32
//      pair per pixel, read from the (L, a, b, w) plane in global memory).
//      The boxes of the candidates are packed in candidate order into the map
//      buffer; a candidate whose box no longer fits walks the plane in global
//      memory instead, with the same per-sample arithmetic and order.
//   3. Pass 1: each warp evaluates its own 64 pixels' previous labels (when
//      they are candidates of the pixel); the previous label usually wins
//      again, and its D stays in the thread's registers.
//   4. Pass 2: each warp checks its pixels against the other candidates
//      whose rectangle (the tile's pixels inside the window) holds them.  A
//      pair whose lower bound fl(fl(lam*d_c(p)) + fl(m^2/r^2*d_s)) exceeds
//      the pixel's pass-1 D cannot win or tie (its computed D is never below
//      the bound) and is not walked; the others are queued per warp and
//      walked 32 at a time by that warp.
//   5. Each walk follows the pixel's path to the candidate's endpoint (one
//      8-byte map load and one packed two-float add per sample), forms D
//      (Eq. 1-3) and takes a 64-bit shared-memory atomicMin of (D bits,
//      candidate slot) for its pixel; slots are in cluster order, so ties go
//      to the smallest k.  The argmin is that of evaluating every pair.
//   6. Each thread writes its pixels' labels; warp-aggregated integer sums of
//      (1, x, y, L, a, b) per label go to the global cluster sums as
//      fire-and-forget reductions.
// The tile body is in scalp_assign_tile.cuh (shared with the persistent
// batched kernel).
// A tile with more candidates than shared memory holds evaluates its pixels
// one by one from the global candidate list instead.
#include <algorithm>
#include <cfloat>
#include <climits>

#include "scalp_launch.h"
#include "scalp_assign_tile.cuh"

namespace scalp {

size_t assign_smem_bytes(int map_cap)
{
    return tile_layout(MAX_TILE_CANDIDATES).maps + (size_t)map_cap * sizeof(float2);
}

// Map capacity (pairs) when ASSIGN_CTAS_PER_SM CTAs share an SM's shared memory.
int assign_map_capacity(int device)
{
    int per_sm = 0, per_cta_max = 0, reserved = 0;
    if (cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&per_cta_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, device) !=
            cudaSuccess)
        return 0;
    // PERSIST_STATIC_SMEM stays free for the persistent batched kernel's own
    // static shared memory (the same capacity serves every assignment kernel)
    long long per_cta = std::min((long long)per_cta_max,
                                 (long long)per_sm / ASSIGN_CTAS_PER_SM - reserved) - PERSIST_STATIC_SMEM;
    per_cta &= ~15LL;
    const long long cap = (per_cta - (long long)tile_layout(MAX_TILE_CANDIDATES).maps) / (long long)sizeof(float2);
    return cap > 0 ? (int)cap : 0;
}

// A grid that leaves SMs without a second tile is bound by the time of one
// tile: with 1024 threads (a pixel each, one CTA per SM) its chain of map
// strips, walks and sums is half as long.  96 x 160 (15 tiles): WIDE_US.
// Above one tile per SM two 512-thread CTAs share an SM instead.
constexpr int ASSIGN_WIDE_THREADS = 1024;
constexpr int ASSIGN_WIDE_TILES = 152;  // SMs

template <typename T, bool COUNT, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == ASSIGN_THREADS ? ASSIGN_CTAS_PER_SM : 1) k_assign(SolveArgs a)
{
    pdl_wait();
    pdl_release();
    extern __shared__ __align__(16) unsigned char smem[];
    assign_tile<T, false, COUNT, THREADS>(a, blockIdx.x, smem);
}

// All tiles of all images of a batch in one launch: block g is tile
// g - tile_base[i] of image i, tile_base being the prefix of tile counts.
template <typename T, bool COUNT>
__global__ void __launch_bounds__(ASSIGN_THREADS, ASSIGN_CTAS_PER_SM) k_assign_batch(BatchArgs b)
{
    pdl_wait();
    pdl_release();
    extern __shared__ __align__(16) unsigned char smem[];
    const int g = blockIdx.x;
    const int i = batch_find(b.tile_base, b.count, g);
    assign_tile<T, true, COUNT>(b.args[i], g - b.tile_base[i], smem);
}

template <typename T, bool COUNT>
static void launch_assign_as(const SolveArgs &a, size_t smem_bytes, cudaStream_t st, bool pdl)
{
    const int tiles = a.n_tx * a.n_ty;
    if (tiles <= ASSIGN_WIDE_TILES)
        pdl_launch(pdl, k_assign<T, COUNT, ASSIGN_WIDE_THREADS>, dim3(tiles), dim3(ASSIGN_WIDE_THREADS), smem_bytes, st, a);
    else
        pdl_launch(pdl, k_assign<T, COUNT, ASSIGN_THREADS>, dim3(tiles), dim3(ASSIGN_THREADS), smem_bytes, st, a);
}

void launch_assign(const SolveArgs &a, int storage, size_t smem_bytes, cudaStream_t st, bool pdl)
{
    if (storage == 0) {
        if (a.count_samples) launch_assign_as<float4, true>(a, smem_bytes, st, pdl);
        else launch_assign_as<float4, false>(a, smem_bytes, st, pdl);
    } else {
        if (a.count_samples) launch_assign_as<uint2, true>(a, smem_bytes, st, pdl);
        else launch_assign_as<uint2, false>(a, smem_bytes, st, pdl);
    }
}

template <typename T, bool COUNT>
static void launch_assign_batch_as(const BatchArgs &b, int total_tiles, size_t smem_bytes, cudaStream_t st, bool pdl)
{
    pdl_launch(pdl, k_assign_batch<T, COUNT>, dim3(total_tiles), dim3(ASSIGN_THREADS), smem_bytes, st, b);
}

void launch_assign_batch(const BatchArgs &b, int storage, bool count, int total_tiles, size_t smem_bytes,
                         cudaStream_t st, bool pdl)
{
    if (total_tiles <= 0) return;
    if (storage == 0) {
        if (count) launch_assign_batch_as<float4, true>(b, total_tiles, smem_bytes, st, pdl);
        else launch_assign_batch_as<float4, false>(b, total_tiles, smem_bytes, st, pdl);
    } else {
        if (count) launch_assign_batch_as<uint2, true>(b, total_tiles, smem_bytes, st, pdl);
        else launch_assign_batch_as<uint2, false>(b, total_tiles, smem_bytes, st, pdl);
    }
}

// Whether the pruning bound's error estimate holds (scalp_assign_tile.cuh):
// coordinates exact in FP32, and lam and m^2/r^2 far enough from both ends of
// the FP32 range that no product under- or overflows where D would not.
bool bound_valid(int H, int W, float lam, float ms2)
{
    return std::max(H, W) <= (1 << 24) && ms2 >= 1e-12f && ms2 <= 1e12f && (lam == 0.0f || lam >= 1e-12f);
}

// The limit is a property of the kernel, shared by every context on the
// device: it is always set to the full map buffer, which covers any launch.
static cudaError_t configure(const void *f)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)assign_smem_bytes(assign_map_capacity(dev)));
}

// (the kernels with and without counting, in both widths)
template <typename T, bool COUNT>
static cudaError_t configure_as(bool batch)
{
    if (batch) return configure((const void *)k_assign_batch<T, COUNT>);
    const cudaError_t e = configure((const void *)k_assign<T, COUNT, ASSIGN_THREADS>);
    return e != cudaSuccess ? e : configure((const void *)k_assign<T, COUNT, ASSIGN_WIDE_THREADS>);
}

template <typename T>
static cudaError_t configure_pair(bool batch)
{
    const cudaError_t e = configure_as<T, false>(batch);
    return e != cudaSuccess ? e : configure_as<T, true>(batch);
}

cudaError_t assign_batch_configure(int storage)
{
    return storage == 0 ? configure_pair<float4>(true) : configure_pair<uint2>(true);
}

cudaError_t assign_configure(int storage)
{
    return storage == 0 ? configure_pair<float4>(false) : configure_pair<uint2>(false);
}

}  // namespace scalp
