// scalp_assign.cu -- the assignment step of SCALP (Algorithm 1, inner loops)
// restated per tile of pixels, plus the fused partial sums of the update.
//
// Algorithm 1 loops over clusters and, for each pixel of a cluster's
// (2r+1)x(2r+1) window, keeps the cluster with the smallest D(p, C_k) (Eq. 3)
// under a strict '<' in ascending k.  Here each pixel evaluates the same set of
// clusters (those whose window holds it, from its tile's candidate list) and
// keeps the smallest (D, k) pair: the same result, in any evaluation order.
//
// One CTA of 512 threads (two per SM) labels a 32 x 32 tile (for grids of few
// tiles: 1024 threads, or 256 on a 16 x 16 tile):
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
//      pair whose lower bound lam*d_c(p) + m^2/r^2*d_s (a dot product of
//      pixel and candidate terms, less a margin for its rounding) exceeds the
//      pixel's pass-1 D cannot win or tie and is not walked; the others are
//      queued per warp and walked 32 at a time by that warp.
//   5. Each walk follows the pixel's path to the candidate's endpoint (one
//      8-byte map load and one packed two-float add per sample), forms D
//      (Eq. 1-3) and takes a 64-bit shared-memory atomicMin of (D bits,
//      candidate slot) for its pixel; slots are in cluster order, so ties go
//      to the smallest k.  The argmin is that of evaluating every pair.
//   6. Each thread writes its pixels' labels; warp-aggregated integer sums of
//      (1, x, y, L, a, b) per label go to the global cluster sums as
//      fire-and-forget reductions.
// Bound: instruction issue (65-68% of the slots; 93.6 M warp instructions on
// 1080 x 1920 with 2000 clusters) and, between its phases, the dependent loads
// of the set-up and the block barriers, at two CTAs of 64 registers a thread.
// With the dot-product bound, tile-relative walks and the map build in strips a
// launch takes 121.2 us there (139.0 before; FP16 planes of 1361 x 2047, step
// 15: 142 from 179; 2160 x 3840 with 10,000 clusters: 447 from 525).
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

// Dynamic shared memory of a CTA with map_cap distance-map pairs.
size_t assign_smem_bytes(int map_cap, int side)
{
    const uint32_t maps = side == TILE_SIDE ? tile_layout<TILE_SIDE>(MAX_TILE_CANDIDATES).maps
                                            : tile_layout<TILE_SIDE_SMALL>(MAX_TILE_CANDIDATES).maps;
    return maps + (size_t)map_cap * sizeof(float2);
}

// Map capacity (pairs) when `ctas` CTAs share an SM's shared memory.
static int map_capacity(int device, int ctas, int side)
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
    long long per_cta = std::min((long long)per_cta_max, (long long)per_sm / ctas - reserved) - PERSIST_STATIC_SMEM;
    per_cta &= ~15LL;
    const long long cap = (per_cta - (long long)assign_smem_bytes(0, side)) / (long long)sizeof(float2);
    return cap > 0 ? (int)cap : 0;
}

constexpr int SMS = 152;

// Small tiles leave as much shared memory to a CTA as the grid's CTAs per SM
// allow, between three and four of them.  (With two, 300 tiles filled every
// SM's shared memory, and the next kernels were placed late: a 240 x 320 solve
// 313 us against 279.)
int assign_map_capacity(int device, int side, int tiles)
{
    const int ctas = side == TILE_SIDE ? ASSIGN_CTAS_PER_SM
                                       : std::min(std::max((tiles + SMS - 1) / SMS, 3), 4);
    return map_capacity(device, ctas, side);
}

// Whether a single image takes small tiles.  A 32 x 32 tile is about 47,000 warp
// instructions, 6 us of an SM at best, so an image of few tiles waits for one
// SM's work while others idle.  Quarter tiles cost a fifth more in all (each
// reads its candidates and builds its maps for 256 pixels) but spread: solves
// of 96 x 160 274 -> 229 us, 200 x 300 290 -> 263, 240 x 320 291 -> 279,
// 321 x 481 357 -> 337, 360 x 480 (180 tiles) 373 -> 362; from 208 tiles on they
// are no faster (400 x 500 386 -> 385 and 377 -> 393, 448 x 512 386 -> 398).
// Above r = 24 a small tile's boxes outgrow its map buffer.
bool small_tiles(int H, int W, double r)
{
    const long long tiles = ceil_div_ll(W, TILE_SIDE) * ceil_div_ll(H, TILE_SIDE);
    return tiles <= 192 && r <= 24.0;
}

// A grid that leaves SMs without a second tile is bound by the time of one
// tile: with 1024 threads (a pixel each, one CTA per SM) its chain of map
// strips, walks and sums is half as long.  Above one tile per SM two
// 512-thread CTAs share an SM instead.
constexpr int ASSIGN_WIDE_THREADS = 1024, ASSIGN_SMALL_THREADS = 256;

template <typename T, bool COUNT, int THREADS, int SIDE>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_assign(SolveArgs a)
{
    pdl_wait();
    pdl_release();
    extern __shared__ __align__(16) unsigned char smem[];
    // a grid of the image's tiles, or (more rows of them than a grid can have)
    // one row of all
    const int tile = (int)(blockIdx.y * gridDim.x + blockIdx.x);
    const bool flat = gridDim.x != (unsigned)a.n_tx;
    assign_tile<T, false, COUNT, THREADS, SIDE>(a, tile, flat ? tile % a.n_tx : (int)blockIdx.x,
                                                flat ? tile / a.n_tx : (int)blockIdx.y, smem);
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
    const int i = batch_find_warp(b.tile_base, b.count, g);
    // The image's arguments in shared memory: in global memory every use was a
    // load on the way to another one (and again after every store), five or
    // six in a row before the tile's first candidate.  64 images, FP32: 2747 us
    // a launch with them there, 2660 as a local copy (which spills), 2575 so;
    // 2787 with a thread's binary search for the image instead of a warp's.
    __shared__ SolveArgs a;
    static_assert(sizeof(SolveArgs) % 4 == 0 && sizeof(SolveArgs) / 4 <= ASSIGN_THREADS, "a word per thread");
    if (threadIdx.x < sizeof(SolveArgs) / 4)
        reinterpret_cast<int *>(&a)[threadIdx.x] = reinterpret_cast<const int *>(&b.args[i])[threadIdx.x];
    __syncthreads();
    const int tile = g - b.tile_base[i];
    assign_tile<T, true, COUNT>(a, tile, tile % a.n_tx, tile / a.n_tx, smem);
}

template <typename T, bool COUNT>
static void launch_assign_as(const SolveArgs &a, size_t smem_bytes, cudaStream_t st, bool pdl)
{
    const int tiles = a.n_tx * a.n_ty;
    const auto launch = [&](auto kernel, int threads) {
        pdl_launch(pdl, kernel, a.n_ty <= 65535 ? dim3(a.n_tx, a.n_ty) : dim3(tiles), dim3(threads), smem_bytes, st, a);
    };
    if (1 << a.tile_shift == TILE_SIDE_SMALL)
        launch(k_assign<T, COUNT, ASSIGN_SMALL_THREADS, TILE_SIDE_SMALL>, ASSIGN_SMALL_THREADS);
    else if (tiles <= SMS)
        launch(k_assign<T, COUNT, ASSIGN_WIDE_THREADS, TILE_SIDE>, ASSIGN_WIDE_THREADS);
    else
        launch(k_assign<T, COUNT, ASSIGN_THREADS, TILE_SIDE>, ASSIGN_THREADS);
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

// The limit is a property of the kernel, shared by every context on the
// device: it is always set to the largest map buffer, which covers any launch.
static cudaError_t configure(const void *f, int side)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)assign_smem_bytes(assign_map_capacity(dev, side, 1), side));
}

// (the kernels with and without counting, in every form)
template <typename T, bool COUNT>
static cudaError_t configure_as(bool batch)
{
    if (batch) return configure((const void *)k_assign_batch<T, COUNT>, TILE_SIDE);
    cudaError_t e = configure((const void *)k_assign<T, COUNT, ASSIGN_THREADS, TILE_SIDE>, TILE_SIDE);
    if (e == cudaSuccess) e = configure((const void *)k_assign<T, COUNT, ASSIGN_WIDE_THREADS, TILE_SIDE>, TILE_SIDE);
    if (e == cudaSuccess)
        e = configure((const void *)k_assign<T, COUNT, ASSIGN_SMALL_THREADS, TILE_SIDE_SMALL>, TILE_SIDE_SMALL);
    return e;
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
