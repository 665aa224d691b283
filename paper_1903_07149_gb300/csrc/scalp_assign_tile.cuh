// scalp_assign_tile.cuh -- the assignment of one tile (32 x 32 or 16 x 16; Algorithm 1's
// inner loops restated per tile, with the fused partial sums of the update):
// the body shared by the per-iteration assignment kernels (scalp_assign.cu)
// and the persistent batched kernel (scalp_persistent.cu).
#pragma once

#include <cfloat>
#include <climits>

#include "scalp_internal.cuh"

namespace scalp {

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// One FP32 pair of a distance map, by 32-bit shared-memory byte address: the
// two floats' bits in one 64-bit word (d_c low).
__device__ __forceinline__ unsigned long long lds_pair_bits(uint32_t addr)
{
    unsigned long long v;
    asm volatile("ld.shared.b64 %0, [%1];" : "=l"(v) : "r"(addr));
    return v;
}

// Both running sums of a walk advanced at once: (d_c, w) += pair, each half
// an FP32 addition rounded to nearest (the same result as two scalar adds).
__device__ __forceinline__ void add_pair(unsigned long long &acc, unsigned long long v)
{
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(v));
}

// Path of Eq. 1 and Eq. 2 between tile pixel (X, Y) and the endpoint (ex, ey)
// over a distance map: places count from the tile's corner, which lies at
// shared-memory address `at` (it may lie outside the map), rows are p8 bytes
// apart.  Yields d_c of the pixel itself and the sums over the path, the same
// samples in the same order and with the same FP32 additions as path_sums()
// over the plane; returns |P|.  The walk starts at the lexicographically
// smaller end, the sign of dx * 2^16 + dy (a map's sides are far below 2^15:
// its rows hold at least four pairs).
__device__ __forceinline__ int path_sums_map(uint32_t at, int p8, int X, int Y, int ex, int ey, float &dcp,
                                             float &sum_dc, float &sum_w)
{
    const uint32_t own = at + (uint32_t)(Y * p8 + X * 8);
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(dcp) : "r"(own));
    const int dx = ex - X, dy = ey - Y, key = dx * 65536 + dy;
    const int adx = abs(dx), ady = abs(dy);
    const bool xmajor = adx >= ady;
    PathSetup s;  // (its steps and slope)
    s.ns = max(adx, ady);
    s.dmin = min(adx, ady);
    const int ys = (dy ^ key) < 0 ? -p8 : p8;  // y falls along the walk, or rises
    const int smaj = xmajor ? 8 : ys, smin = xmajor ? ys : 8;
    const uint32_t q0 = key < 0 ? at + (uint32_t)(ey * p8 + ex * 8) : own;
    unsigned long long acc = 0;  // (+0.0f, +0.0f)
    const auto visit = [&](uint32_t q) { add_pair(acc, lds_pair_bits(q)); };
    // the fixed-point forms of the steps (fewer instructions per sample)
    // cover every path of up to FIXED_STEP_MAX_NS steps
    const int len = s.ns <= FIXED_STEP_MAX_NS ? walk_grouped<4>(q0, smaj, smin, s, visit)
                                              : walk_with<ErrorTermStep>(q0, smaj, smin, s, visit);
    sum_dc = __uint_as_float((unsigned)acc);
    sum_w = __uint_as_float((unsigned)(acc >> 32));
    return len;
}

// Shared-memory layout; every section starts on a 16-byte boundary (int4
// loads and 8-byte atomics need it).  The fixed sections come first; the
// per-candidate records follow, sized for the tile's own candidate count, and
// the distance maps fill the rest (a tile with few candidates has more room).
__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }
// Pairs the warps' queues of a tile hold together (pass 2): 2.5 a pixel.
__host__ __device__ constexpr int assign_queues(int side) { return side * side * 5 / 2; }
template <int SIDE>
struct AssignSmem {
    static constexpr size_t best = 0;
    static constexpr size_t queue = align16(best + SIDE * SIDE * sizeof(unsigned long long));
    static constexpr size_t misc = align16(queue + assign_queues(SIDE) * sizeof(uint16_t));
    static constexpr size_t records = align16(misc + 64);
};
// Per candidate (rank c): three 16-byte records the walk reads,
//   rec0 = (columns, rows, K bits, g_y bits)         its rectangle as a mask of
//          the tile's columns and one of its rows; terms of the bound
//   rec1 = (ex, ey, xk bits, yk bits)                endpoint, X_k
//   rec2 = (endpoint from the tile's corner, address of that corner on the
//          map, bytes per map row, or 0: walk the plane)
// the map box for the build, box = (bx0, by0, pitch, width | height << 16),
// the colour C_k, col = (l_k, a_k, b_k, g_x), the cluster index
// cid, the box area and the prefixes mfirst and cfirst of the map layout.
struct TileLayout {
    uint32_t rec0, rec1, rec2, box, col, cid, area, mfirst, cfirst, maps;
};
template <int SIDE>
__host__ __device__ constexpr TileLayout tile_layout(int n)
{
    TileLayout t{};
    t.rec0 = (uint32_t)AssignSmem<SIDE>::records;
    t.rec1 = t.rec0 + (uint32_t)n * 16u;
    t.rec2 = t.rec1 + (uint32_t)n * 16u;
    t.box = t.rec2 + (uint32_t)n * 16u;
    t.col = t.box + (uint32_t)n * 16u;
    t.cid = t.col + (uint32_t)n * 16u;
    t.area = (uint32_t)align16(t.cid + (size_t)n * 4);
    t.mfirst = (uint32_t)align16(t.area + (size_t)n * 4);
    t.cfirst = (uint32_t)align16(t.mfirst + (size_t)(n + 1) * 4);
    t.maps = (uint32_t)align16(t.cfirst + (size_t)(n + 1) * 4);
    return t;
}
// The map pairs a tile of n candidates has beyond the capacity sized for
// MAX_TILE_CANDIDATES.
template <int SIDE>
__host__ __device__ constexpr int extra_map_pairs(int n)
{
    return (int)((tile_layout<SIDE>(MAX_TILE_CANDIDATES).maps - tile_layout<SIDE>(n).maps) / 8u);
}
static_assert(MAX_TILE_CANDIDATES % 32 == 0, "the scans give each lane whole candidates");

// Rank of cluster k among the tile's candidates (cid sorted ascending), or -1.
__device__ __forceinline__ int find_slot(const int *cid, int cnt, int k)
{
    int lo = 0, hi = cnt;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (cid[mid] < k) lo = mid + 1;
        else hi = mid;
    }
    return lo < cnt && cid[lo] == k ? lo : -1;
}

// The pruning bound.  With q = lam |v - c|^2 + m^2/r^2 |X - X_k|^2 (v, X the
// pixel's own sample and place), the D that scalp_distance() computes is at
// least q up to rounding: the path term of Eq. 1 and the contour term of
// Eq. 2 are non-negative and every factor is at least one.  Expanded,
//   q = P(pixel) + K(cluster) + f . g,
//   P = lam |v|^2 + m^2/r^2 |X|^2,  f = (-2 lam v, X),
//   K = lam |c|^2 + m^2/r^2 |X_k|^2,  g = (c, -2 m^2/r^2 X_k)
// with X and X_k from the tile's corner: five multiply-adds per pair, against
// fourteen operations for the two squared distances.  P and K are scaled by
// 1 - 2^-17 here.  With u = 2^-24, the rounding of K (8 u K), of f and g (3 u
// |f . g|) and of the chain (10 u (P + K)) adds up to less than 30 u (P + K)
// as |f . g| <= P + K, so P' + K' + f . g stays below q - 98 u (P + K); the
// computed D is above q - 20 u (P + K) (at most ten roundings).  A pair whose
// bound exceeds the pixel's pass-1 D raised by 2^-20 (bound_threshold()
// subtracts P') therefore has a larger D: it can neither win nor tie.
// That holds for every accepted weight, and for sides up to 2^24, whose places
// FP32 holds exactly (the host turns the pruning off above):
//   * Products below the normal range err by 2^-150 each, at most twenty of
//     them, times places and samples below 2^7: D is raised by 2^-100 as well.
//   * P or D above 1e30 prunes nothing.  K then overflows only where q does not
//     stay below 1e30 (|f . g| <= 2 sqrt(P K)), and a NaN prunes nothing.
// BOUND_SCALE and bound_threshold() are in scalp_internal.cuh (the supervoxels
// use them too).

__device__ __forceinline__ unsigned long long pack_best(float D, int slot)
{
    // D >= 0, so its IEEE bits order like the value; ties fall to the slot
    return ((unsigned long long)__float_as_uint(D) << 32) | (unsigned)slot;
}

// The map layout by one warp: mfirst = exclusive prefix of the box areas
// (cnt + 1 entries); the leading candidates whose boxes end within cap get a
// map, of BUILD_STRIP-column strips whose prefix goes to cfirst (cnt + 1
// entries; none for the others).  Returns the map entries used.
constexpr int BUILD_STRIP = 8;
__device__ __forceinline__ int warp_scan_maps(const int *area, const int4 *box, int *mfirst, int *cfirst, int cnt,
                                              int cap, int lane)
{
    constexpr int PER = MAX_TILE_CANDIDATES / 32;
    int v[PER], ch[PER], sum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int c = lane * PER + i;
        v[i] = c < cnt ? area[c] : 0;
        sum += v[i];
    }
    int incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    // a box fits when its prefix end is within cap (the ends only grow)
    int run = incl - sum, fit = 0, csum = 0;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int c = lane * PER + i;
        if (c < cnt) mfirst[c] = run;
        run += v[i];
        const bool mapped = c < cnt && v[i] > 0 && run <= cap;
        if (c < cnt && run <= cap) fit = run;
        ch[i] = mapped ? ((box[c].w & 0xffff) + BUILD_STRIP - 1) / BUILD_STRIP : 0;
        csum += ch[i];
    }
    if (lane == 31) mfirst[cnt] = incl;
    int cincl = csum;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, cincl, o);
        if (lane >= o) cincl += t;
    }
    int crun = cincl - csum;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int c = lane * PER + i;
        if (c < cnt) cfirst[c] = crun;
        crun += ch[i];
    }
    if (lane == 31) cfirst[cnt] = cincl;
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)fit);
}

// One tile of one image (the body shared by the single-image and the batched
// kernels), SIDE x SIDE pixels by THREADS threads.  The pixels of a candidate's
// window that lie in the tile form a rectangle; each warp owns one or two
// blocks of 8 x 4 pixels of the tile (column tx, row ty of the image's tiles).
// PREFETCH_TILE: the tile's plane rows are first asked into L2 (for batches,
// whose planes outgrow L2; an image whose plane stays in L2 only pays for it).
// COUNT: the work is counted when a.count_samples asks for it (the counting
// code costs the walks and the bound even when it is off).
template <typename T, bool PREFETCH_TILE = false, bool COUNT = true, int THREADS = ASSIGN_THREADS, int SIDE = TILE_SIDE>
__device__ __forceinline__ void assign_tile(const SolveArgs &a, int tile, int tx, int ty, unsigned char *smem)
{
    constexpr int PIX_PER_THREAD = SIDE * SIDE / THREADS;
    constexpr int WARPS = THREADS / 32;
    constexpr int QUEUE = assign_queues(SIDE) / WARPS;  // pairs a warp's queue holds
    constexpr int BUILD_UNROLL = STRIP_ROWS;  // samples per lane in flight
    const T *__restrict__ plane = reinterpret_cast<const T *>(
        sizeof(T) == 16 ? (const void *)a.plane32 : (const void *)a.plane16);
    const int x0 = tx * SIDE, y0 = ty * SIDE;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    unsigned long long *best = reinterpret_cast<unsigned long long *>(smem + AssignSmem<SIDE>::best);
    int *misc = reinterpret_cast<int *>(smem + AssignSmem<SIDE>::misc);

    // this thread's pixels: block (warp * PIX_PER_THREAD + j) of the tile
    // (a warp's blocks lie side by side), lane within it
    auto my_pixel = [&](int j, int &qx, int &qy) {
        const int blk = warp + j * WARPS;
        qx = x0 + (blk % (SIDE / WARP_BLOCK_X)) * WARP_BLOCK_X + (lane % WARP_BLOCK_X);
        qy = y0 + (blk / (SIDE / WARP_BLOCK_X)) * WARP_BLOCK_Y + (lane / WARP_BLOCK_X);
    };

    const int off = a.tile_off[tile];
    // the list capacity is a proven bound; the held_lamp only guards memory if the
    // device-side overflow check (reported as an error) ever fired
    const int cnt = (int)max(0LL, min((long long)a.tile_off[tile + 1], a.tile_cap) - off);
    const bool fast = cnt <= MAX_TILE_CANDIDATES;
    // the records for this tile's candidates, then its maps
    const TileLayout lay = tile_layout<SIDE>(fast ? cnt : 0);
    int4 *rec0 = reinterpret_cast<int4 *>(smem + lay.rec0);
    int4 *rec1 = reinterpret_cast<int4 *>(smem + lay.rec1);
    int4 *rec2 = reinterpret_cast<int4 *>(smem + lay.rec2);
    int4 *box = reinterpret_cast<int4 *>(smem + lay.box);
    float4 *col = reinterpret_cast<float4 *>(smem + lay.col);
    int *cid = reinterpret_cast<int *>(smem + lay.cid);
    int *area = reinterpret_cast<int *>(smem + lay.area);
    int *mfirst = reinterpret_cast<int *>(smem + lay.mfirst);
    int *cfirst = reinterpret_cast<int *>(smem + lay.cfirst);
    const uint32_t maps_u32 = smem_u32(smem + lay.maps);
    float2 *maps = reinterpret_cast<float2 *>(smem + lay.maps);
    const int map_cap = a.map_cap > 0 ? a.map_cap + extra_map_pairs<SIDE>(fast ? cnt : 0) : 0;
    if (tid == 0) {  // this tile's list is read: ready the counts for the next update
        a.tile_count[tile] = 0;
        a.tile_cursor[tile] = 0;
        // the last projection (and lists) completed before this launch: its
        // queue starts again for the next update
        if (tile == 0) a.ctr->nproj = 0;
    }

    // the tile's plane rows into L2 while the set-up runs, so that the map
    // build finds them there (x0 * sizeof(T) and the row pitch are multiples
    // of 16 bytes, and so is every row's length: the bulk prefetch's rules)
    static_assert(SIDE <= 32, "one row per lane");
    if (PREFETCH_TILE && warp == WARPS - 1) {
        const int rows = min(a.H - y0, SIDE);
        const uint32_t bytes = (uint32_t)(min(SIDE, a.pitch - x0) * (int)sizeof(T));
        if (lane < rows) {
            const T *p = plane + (long long)(y0 + lane) * a.pitch + x0;
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
        }
    }

    // this thread's pixels' previous labels (their loads overlap the set-up)
    int prev_lab[PIX_PER_THREAD];
#pragma unroll
    for (int j = 0; j < PIX_PER_THREAD; ++j) {
        int px, py;
        my_pixel(j, px, py);
        prev_lab[j] = fast && px < a.W && py < a.H ? a.labels[(long long)py * a.W + px] : -1;
    }
    // the samples of this thread's pixels
    const auto load_own = [&](T (&own)[PIX_PER_THREAD]) {
#pragma unroll
        for (int j = 0; j < PIX_PER_THREAD; ++j) {
            int px, py;
            my_pixel(j, px, py);
            own[j] = px < a.W && py < a.H ? __ldg(plane + (long long)py * a.pitch + px) : T{};
        }
    };
    if (tid == 0) {
        misc[4] = 0;  // path samples and pairs (counting on)
        misc[5] = 0;
    }
    // the records of candidate id (rank among the tile's sorted ids)
    const auto write_records = [&](int rank, int id, const ClusterDev &cd) {
        cid[rank] = id;
        // window x tile (clipped to the image)
        const int xa = max(cd.xlo, x0), xb = min(min(cd.xhi, x0 + SIDE - 1), a.W - 1);
        const int ya = max(cd.ylo, y0), yb = min(min(cd.yhi, y0 + SIDE - 1), a.H - 1);
        const int w = max(xb - xa + 1, 0), h = max(yb - ya + 1, 0);
        static_assert(SIDE <= 32, "a rectangle is two 32-bit masks");
        const bool some = w > 0 && h > 0;
        const float kx = cd.xk - (float)x0, ky = cd.yk - (float)y0;
        const float K = BOUND_SCALE * fmaf(a.lam, fmaf(cd.L, cd.L, fmaf(cd.a, cd.a, cd.b * cd.b)),
                                           a.ms2 * fmaf(kx, kx, ky * ky));
        rec0[rank] = make_int4(some ? (int)((0xffffffffu >> (32 - w)) << (xa - x0)) : 0,
                               some ? (int)((0xffffffffu >> (32 - h)) << (ya - y0)) : 0, __float_as_int(K),
                               __float_as_int(-2.0f * a.ms2 * ky));
        rec1[rank] = make_int4(cd.ex, cd.ey, __float_as_int(cd.xk), __float_as_int(cd.yk));
        col[rank] = make_float4(cd.L, cd.a, cd.b, -2.0f * a.ms2 * kx);
        // map box: the rectangle and the endpoint (both inside the image).
        // Rows are padded to a pitch = 4 (mod 8) pairs: the walks of a warp
        // then spread over the shared-memory banks (neighbouring rows start
        // 8 banks apart).  A mapped box has width and height below 2^16 (its
        // pitch is at least 4, its area at most the buffer's).
        int bx0 = 0, by0 = 0, pitch = 4, size = 0;
        long long n = 0;
        if (some) {
            bx0 = min(xa, cd.ex);
            by0 = min(ya, cd.ey);
            const int bw = max(xb, cd.ex) - bx0 + 1, bh = max(yb, cd.ey) - by0 + 1;
            pitch = bw + ((4 - bw) & 7);
            n = (long long)pitch * bh;
            size = min(bw, 0xffff) | (min(bh, 0xffff) << 16);
        }
        box[rank] = make_int4(bx0, by0, pitch, size);
        // a box larger than the whole buffer never fits: held_lamp it so that the
        // prefix sums stay small
        area[rank] = map_cap > 0 ? (int)min(n, (long long)map_cap + 1) : 0;
    };
    // the candidates sorted by cluster index (ranks of distinct ids), their
    // records and the map layout; each warp readies its own pixels' best words
    if (fast && cnt <= 32) {
        // one warp: ranks by shuffles, no block barrier until the layout is done
        if (warp == 0) {
            int myid = INT_MAX;
            ClusterDev cd;
            if (lane < cnt) {
                myid = a.tile_list[off + lane];
                cd = a.cdev[myid];
            }
            int rank = 0;
            for (int j = 0; j < 32; ++j) rank += __shfl_sync(0xffffffffu, myid, j) < myid;
            if (lane < cnt) write_records(rank, myid, cd);
            __syncwarp();
            const int used = warp_scan_maps(area, box, mfirst, cfirst, cnt, map_cap, lane);
            if (lane == 0) misc[2] = used;
        }
#pragma unroll
        for (int j = 0; j < PIX_PER_THREAD; ++j) {
            int px, py;
            my_pixel(j, px, py);
            best[(py - y0) * SIDE + (px - x0)] = ~0ull;
        }
    } else {
        // the id staging reuses the `best` words before they are initialised
        int *ids = reinterpret_cast<int *>(best);
        int myid = INT_MAX;
        ClusterDev cd;  // this thread's candidate: its load overlaps the barrier
        if (fast && tid < cnt) {
            myid = a.tile_list[off + tid];
            ids[tid] = myid;
            cd = a.cdev[myid];
        }
        __syncthreads();
        if (fast && tid < cnt) {
            int rank = 0;
            for (int j = 0; j < cnt; ++j) rank += ids[j] < myid;
            write_records(rank, myid, cd);
        }
        __syncthreads();
        for (int i = tid; i < SIDE * SIDE; i += THREADS) best[i] = ~0ull;
        if (warp == 0 && fast) {
            const int used = warp_scan_maps(area, box, mfirst, cfirst, cnt, map_cap, lane);
            if (lane == 0) misc[2] = used;
        }
    }
    __syncthreads();

    // each pixel's previous label, as a candidate slot when the pixel lies in
    // that candidate's rectangle (-1 otherwise): pass 1 below evaluates it
    // first, pass 2 skips it
    int slot[PIX_PER_THREAD];
#pragma unroll
    for (int j = 0; j < PIX_PER_THREAD; ++j) {
        int px, py;
        my_pixel(j, px, py);
        int c = prev_lab[j] >= 0 ? find_slot(cid, cnt, prev_lab[j]) : -1;
        if (c >= 0) {
            const int4 r0 = rec0[c];
            if (!(((unsigned)r0.x >> (px - x0)) & ((unsigned)r0.y >> (py - y0)) & 1u)) c = -1;
        }
        slot[j] = c;
    }

    // the distance maps of the candidates whose boxes fit: entries [0, used)
    // hold the leading candidates' boxes back to back, row-major (no walk reads
    // the padding columns of a row)
    const int used = fast ? misc[2] : 0;
    if (fast) {
        if (tid < cnt) {
            const int4 b = box[tid];
            const bool mapped = area[tid] > 0 && mfirst[tid + 1] <= used;
            rec2[tid] = make_int4(rec1[tid].x - x0, rec1[tid].y - y0,
                                  (int)(maps_u32 + 8u * (uint32_t)(mfirst[tid] - (b.y - y0) * b.z - (b.x - x0))),
                                  mapped ? b.z * 8 : 0);
        }
        // Warps take the boxes' strips of BUILD_STRIP columns in turn: 8
        // columns x 4 rows of lanes move down the strip, so an entry costs
        // two additions for its places instead of a division by the pitch,
        // and a candidate's record is read once per strip (about nine rows of
        // lanes on HD).  A row of lanes covers rows {0, 2, 1, 3}: the two rows of a half warp
        // then lie 16 banks apart.  Lanes past the box read its last column
        // or row and store nothing.
        const int n_strips = cfirst[cnt];
        const int lrow = ((lane >> 3) & 1) << 1 | lane >> 4, lcol = lane & 7;
        int c = 0;
        for (int g = warp; g < n_strips; g += WARPS) {
            while (g >= cfirst[c + 1]) ++c;
            const int4 b = box[c];
            const float4 ck = col[c];
            const int bw = b.w & 0xffff, bh = (int)((unsigned)b.w >> 16);
            const int cx = (g - cfirst[c]) * BUILD_STRIP + lcol;
            // the box's first pixel
            const T *__restrict__ pbox = plane + (long long)b.y * a.pitch + b.x;
            StripPlaces at = strip_places(lrow, bh, a.pitch, bw, cx);
            float2 *m = maps + (mfirst[c] + lrow * b.z + cx);
            const int mstep = 4 * b.z;
            for (int r = 0; r < bh; r += 4 * BUILD_UNROLL) {
                T v[BUILD_UNROLL];  // raw samples: all loads issue before any use
#pragma unroll
                for (int u = 0; u < BUILD_UNROLL; ++u) v[u] = __ldg(pbox + min(at.off + u * at.step, at.last));
#pragma unroll
                for (int u = 0; u < BUILD_UNROLL; ++u) {
                    const float4 q = sample_value(v[u]);
                    const float2 pair = make_float2(colour_dist(q, ck.x, ck.y, ck.z), q.w);
                    if (at.off < (u == 0 ? at.end : at.more)) *m = pair;
                    at.off += at.step;
                    m += mstep;
                }
            }
        }
    }
    __syncthreads();

    // with counting on, the tile's path samples and pairs are summed in
    // misc[4], misc[5] (zeroed at the start; far below 2^32 per tile)
    unsigned *tile_samples = reinterpret_cast<unsigned *>(misc + 4);
    int bestk[PIX_PER_THREAD];  // per-pixel path only
#pragma unroll
    for (int j = 0; j < PIX_PER_THREAD; ++j) bestk[j] = INT_MAX;

    // D of tile pixel (X, Y) for candidate slot c (Eq. 1-3), its path length
    // in len: on a map when the candidate has one, else on the plane
    auto pair_distance = [&](int X, int Y, int c, int &len) {
        const int4 r2 = rec2[c];
        const float2 xk = *reinterpret_cast<const float2 *>(&rec1[c].z);
        const int qx = x0 + X, qy = y0 + Y;
        const float ddx = (float)qx - xk.x, ddy = (float)qy - xk.y;
        float dcp, sdc, sw;
        if (r2.w != 0) {
            len = path_sums_map((uint32_t)r2.z, r2.w, X, Y, r2.x, r2.y, dcp, sdc, sw);
        } else {
            const float4 ck = col[c];
            const int4 r1 = rec1[c];
            dcp = colour_dist(fetch_sample<T>(plane + (long long)qy * a.pitch + qx), ck.x, ck.y, ck.z);
            len = path_sums<T>(plane, a.pitch, 0, 0, path_setup(qx, qy, r1.x, r1.y), ck.x, ck.y, ck.z, sdc, sw);
        }
        return scalp_distance(dcp, sdc, sw, len, a.lam, a.gamma, a.ms2, fmaf(ddx, ddx, ddy * ddy));
    };
    auto count_pair = [&](int len) {
        if (COUNT && a.count_samples) {
            atomicAdd(tile_samples, (unsigned)len);
            atomicAdd(tile_samples + 1, 1u);
        }
    };

    if (fast) {
        // Pass 1: each pixel's previous label first, when it is a candidate
        // of the pixel (it usually wins again).  Its D bounds the minimum, so
        // pass 2 can skip every candidate whose lower bound exceeds it: such
        // a candidate's D is larger than the minimum and cannot win or tie.
        // The argmin is unchanged.  Each warp walks its own pixels here.
        float dprev[PIX_PER_THREAD];  // D of the previous label; NaN: none
#pragma unroll
        for (int j = 0; j < PIX_PER_THREAD; ++j) dprev[j] = __int_as_float(0x7fffffff);
#pragma unroll 1
        for (int j = 0; j < PIX_PER_THREAD; ++j) {
            int px, py;
            my_pixel(j, px, py);
            int c = slot[0];
#pragma unroll
            for (int i = 1; i < PIX_PER_THREAD; ++i)  // (registers: constant indices)
                if (i == j) c = slot[i];
            if (c >= 0) {
                int len;
                const float D = pair_distance(px - x0, py - y0, c, len);
                best[(py - y0) * SIDE + (px - x0)] = pack_best(D, c);  // (the pixel's first D)
#pragma unroll
                for (int i = 0; i < PIX_PER_THREAD; ++i)
                    if (i == j) dprev[i] = D;
                count_pair(len);
            }
        }
        __syncwarp();  // the D's before the warp's other lanes lower them

        // Pass 2: each warp checks its own pixels against every other
        // candidate whose rectangle holds them, and queues the surviving
        // pairs (slot << 6 | block << 5 | lane); then it walks the queue 32
        // pairs at a time, one per lane.  (A barrier before the walks, to
        // share them among the warps, cost more than the uneven loads it
        // evens out.)  The pixels' samples are at hand only while the queue
        // fills: held across the walks as well they spill registers (FP32, HD
        // 140.0 us a launch against 134.7).
        static_assert(WARPS % (SIDE / WARP_BLOCK_X) == 0, "the warp's blocks lie in one column of blocks");
        static_assert(PIX_PER_THREAD <= 2 && MAX_TILE_CANDIDATES <= 1024, "queued pairs pack into 16 bits");
        static_assert(QUEUE > 32 * PIX_PER_THREAD, "a queue takes a candidate's pairs after a full batch is left over");
        constexpr int ROW_STEP = WARPS / (SIDE / WARP_BLOCK_X) * WARP_BLOCK_Y;  // block 1 lies this far below block 0
        int px, py;
        my_pixel(0, px, py);
        const int bx = px - lane % WARP_BLOCK_X, by = py - lane / WARP_BLOCK_X;
        uint16_t *wq = reinterpret_cast<uint16_t *>(smem + AssignSmem<SIDE>::queue) + warp * QUEUE;
        int queued = 0, c0 = -32;                    // warp-uniform, as all that follows
        unsigned meets[PIX_PER_THREAD] = {}, any = 0;  // candidates c0 + bit left, per block and over both
        for (bool more = true; more;) {
            // the pixels' side of the bound
            float fL[PIX_PER_THREAD], fa[PIX_PER_THREAD], fb[PIX_PER_THREAD], thr[PIX_PER_THREAD];
            const float X = (float)(px - x0);
            float Y[PIX_PER_THREAD];
            {
                T own[PIX_PER_THREAD];
                load_own(own);
#pragma unroll
                for (int j = 0; j < PIX_PER_THREAD; ++j) {
                    const float4 v = sample_value(own[j]);
                    Y[j] = (float)(py - y0 + j * ROW_STEP);
                    thr[j] = a.prune ? bound_threshold(dprev[j], fmaf(a.lam, fmaf(v.x, v.x, fmaf(v.y, v.y, v.z * v.z)),
                                                                      a.ms2 * fmaf(X, X, Y[j] * Y[j])))
                                     : __int_as_float(0x7fffffff);
                    fL[j] = -2.0f * a.lam * v.x;
                    fa[j] = -2.0f * a.lam * v.y;
                    fb[j] = -2.0f * a.lam * v.z;
                }
            }
            const unsigned lanes_below = (1u << lane) - 1u;
            while (queued <= QUEUE - 32 * PIX_PER_THREAD) {
                if (!any) {
                    // the next 32 candidates: which of their rectangles meet
                    // each of the warp's blocks, one candidate per lane
                    c0 += 32;
                    more = c0 < cnt;
                    if (!more) break;
                    const int4 r0 = c0 + lane < cnt ? rec0[c0 + lane] : make_int4(0, 0, 0, 0);
                    const bool mx = ((unsigned)r0.x >> (bx - x0)) & ((1u << WARP_BLOCK_X) - 1u);
#pragma unroll
                    for (int j = 0; j < PIX_PER_THREAD; ++j) {
                        const bool my = ((unsigned)r0.y >> (by - y0 + j * ROW_STEP)) & ((1u << WARP_BLOCK_Y) - 1u);
                        meets[j] = __ballot_sync(0xffffffffu, mx && my);
                        any |= meets[j];
                    }
                    continue;
                }
                const int b = __ffs(any) - 1, c = c0 + b;
                any &= any - 1;
                const int4 r0 = rec0[c];
                const float4 ck = col[c];
                const float base = fmaf(X, ck.w, __int_as_float(r0.z));
                const bool inx = (unsigned)r0.x & (1u << (px - x0));
#pragma unroll
                for (int j = 0; j < PIX_PER_THREAD; ++j) {
                    if (!((meets[j] >> b) & 1u)) continue;
                    // (a pixel of the rectangle lies in the image)
                    const bool in = inx && ((unsigned)r0.y & (1u << (py - y0 + j * ROW_STEP))) && slot[j] != c;
                    const float bound = fmaf(fL[j], ck.x, fmaf(fa[j], ck.y, fmaf(fb[j], ck.z,
                                             fmaf(Y[j], __int_as_float(r0.w), base))));
                    const bool loses = bound > thr[j];
                    if (COUNT && in && loses) {
                        // a pair that cannot win is not walked (counted as the method's work)
                        const int4 r1 = rec1[c];
                        count_pair(max(abs(px - r1.x), abs(py + j * ROW_STEP - r1.y)) + 1);
                    }
                    const bool keep = in && !loses;
                    const unsigned kept = __ballot_sync(0xffffffffu, keep);
                    if (keep) wq[queued + __popc(kept & lanes_below)] = (uint16_t)((c << 6) | (j << 5) | lane);
                    queued += __popc(kept);
                }
            }
            __syncwarp();  // the queued pairs
            int from = 0;
#pragma unroll 1
            for (; more ? from + 32 <= queued : from < queued; from += 32) {
                if (from + lane >= queued) continue;
                const int e = wq[from + lane], c = e >> 6;
                const int X = bx - x0 + (e & 31) % WARP_BLOCK_X;
                const int Y = by - y0 + (e & 31) / WARP_BLOCK_X + ((e >> 5) & 1) * ROW_STEP;
                int len;
                const float D = pair_distance(X, Y, c, len);
                atomicMin(&best[Y * SIDE + X], pack_best(D, c));
                count_pair(len);
            }
            if (more) {  // the pairs left over start the next queue
                queued -= from;
                const uint16_t e = lane < queued ? wq[from + lane] : (uint16_t)0;
                __syncwarp();
                if (lane < queued) wq[lane] = e;
                __syncwarp();
            }
        }
    } else {
        // per-pixel path: every candidate straight from the global list.  The
        // pointers in registers: from the batch's shared memory in each round,
        // 40 small images with step 3 took 8.88 ms per five iterations, 8.43
        // so.  FP16 planes hold the weights as well (or the hot path above is
        // allocated worse: 12 served images 7.21 ms, 7.05 so); with FP32 it is
        // the other way round (batch of 64 28.6 ms, 28.1 so).
        const int *list = a.tile_list + off;
        const ClusterDev *cdev = a.cdev;
        constexpr bool HOLD = sizeof(T) == 8;
        const int held_pitch = a.pitch;
        const float held_lam = a.lam, held_gamma = a.gamma, held_ms2 = a.ms2;
#pragma unroll 1
        for (int j = 0; j < PIX_PER_THREAD; ++j) {
            int px, py;
            my_pixel(j, px, py);
            if (px >= a.W || py >= a.H) continue;
            const float4 own = fetch_sample<T>(plane + (long long)py * (HOLD ? held_pitch : a.pitch) + px);
            float bestD = FLT_MAX;
            for (int i = 0; i < cnt; ++i) {
                const int k = list[i];
                const ClusterDev cd = cdev[k];
                if (px < cd.xlo || px > cd.xhi || py < cd.ylo || py > cd.yhi) continue;
                const PathSetup s = path_setup(px, py, cd.ex, cd.ey);
                float sdc, sw;
                const int len = path_sums<T>(plane, HOLD ? held_pitch : a.pitch, 0, 0, s, cd.L, cd.a, cd.b, sdc, sw);
                const float dcp = colour_dist(own, cd.L, cd.a, cd.b);
                const float ddx = (float)px - cd.xk, ddy = (float)py - cd.yk;
                const float ds = fmaf(ddx, ddx, ddy * ddy);
                const float D = scalp_distance(dcp, sdc, sw, len, HOLD ? held_lam : a.lam,
                                               HOLD ? held_gamma : a.gamma, HOLD ? held_ms2 : a.ms2, ds);
                if (D < bestD || (D == bestD && k < bestk[j])) {
                    bestD = D;
                    bestk[j] = k;
                }
                if (COUNT && a.count_samples) {
                    atomicAdd(tile_samples, (unsigned)len);
                    atomicAdd(tile_samples + 1, 1u);
                }
            }
        }
    }
    // a warp's pixels were walked by that warp alone (both passes, or the
    // per-pixel path), so its lanes' writes to them need only a warp barrier
    __syncwarp();

    // labels and the warp-aggregated integer sums of the update; the
    // pixels' own samples are all requested first
    T own[PIX_PER_THREAD];
    load_own(own);
#pragma unroll
    for (int j = 0; j < PIX_PER_THREAD; ++j) {
        int px, py;
        my_pixel(j, px, py);
        const bool valid = px < a.W && py < a.H;
        const long long p = (long long)py * a.W + px;
        int lab = -1;
        if (valid) {
            if (fast) {
                const unsigned long long b = best[(py - y0) * SIDE + (px - x0)];
                if (b != ~0ull) lab = cid[(int)(b & 0xffffffffu)];
            } else if (bestk[j] != INT_MAX) {
                lab = bestk[j];
            }
            if (lab >= 0) {
                a.labels[p] = lab;
            } else {
                lab = a.labels[p];  // no window reaches p: keep its label
                a.orphan_list[atomicAdd(&a.ctr->orphans, 1)] = (int)p;
            }
        }
        // fire-and-forget reductions into the global cluster sums, one set
        // per label group of the warp (offsets within the tile)
        warp_aggregate_global(valid, lab, x0, y0, px - x0, py - y0, sample_value(own[j]), a.acc);
    }
    if (COUNT && a.count_samples) {
        __syncthreads();  // every warp's counts are in (a CTA-uniform branch)
        if (tid == 0) {
            atomicAdd(&a.ctr->samples, (unsigned long long)tile_samples[0]);
            atomicAdd(&a.ctr->pairs, (unsigned long long)tile_samples[1]);
        }
        // (candidate, tile) rectangles walked on a map and on the plane
        if (tid == 0) {
            unsigned long long on_map = 0, on_plane = 0;
            for (int c = 0; c < cnt; ++c) {
                if (fast && rec0[c].x == 0) continue;  // no pixel
                if (fast && rec2[c].w != 0) ++on_map;
                else ++on_plane;
            }
            atomicAdd(&a.ctr->map_rects, on_map);
            atomicAdd(&a.ctr->plane_rects, on_plane);
        }
    }
}

}  // namespace scalp
