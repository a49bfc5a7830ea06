// Exact outer volume of oriented boxes on the occupancy lattice (Eq. 4).
//
// A box is the integer slab set lo_a <= n_a . (256 p) <= hi_a.  Counting:
//   prep   per box: index-space bounds Lq = ceil(lo / 256), Hq = floor(hi / 256),
//          a conservative (j, k) rectangle (exact integer cofactors, FP32
//          geometry with explicit margins), the row axis (x unless the context
//          counts along the axis of the smallest shadow), the tile shape, the
//          per-row step of each slab's quotient (remainder and 32.32 forms) and
//          three separating bands of the box's shadow on the (j, k) plane; the
//          last block to finish scans the tile counts into per-box offsets and
//          clears the work counter;
//   count  persistent warps take one tile at a time from the counter: wj (y)
//          x wk * tk (z) rows of one box, wj * wk = 32 lanes.  A tile outside
//          the box's shadow is skipped and the rows of a tile are clipped to
//          it.  Each lane owns one j and walks tk rows along z: it divides the
//          lower slab bounds exactly once per tile (integer reciprocal; the
//          upper ones follow from the slabs' widths) and then steps all six as
//          32.32 fixed-point values (boxes whose three slabs are DDA slabs) or
//          with a remainder carry (the general loop), so each row's exact
//          x-interval costs adds and compares only.  The occupied bits of the
//          interval are popcounted over 64-bit words; outer volume = interval
//          length - occupied bits, and rows or points outside [0, N)^3 are all
//          empty.
// Counts are integer sums (warp reduction + one 64-bit atomic per tile), so
// the result does not depend on scheduling.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "counting.cuh"
#include "internal.h"

#ifndef OBB_GRAB
#define OBB_GRAB 1
#endif
// OBB_COUNT_MINB, OBB_COUNT_MINB_SMALL: resident blocks of the counting kernel
// per SM the register budget aims at, on lattices of at least
// OBB_ORDER_MIN_MB MiB and on smaller ones
#ifndef OBB_COUNT_MINB
#define OBB_COUNT_MINB 5
#endif
#ifndef OBB_COUNT_MINB_SMALL
#define OBB_COUNT_MINB_SMALL 4
#endif
// OBB_ORDER_MIN_BOXES, OBB_ORDER_MIN_MB: batches of at least this many boxes on
// lattices of at least this many MiB of occupancy words are counted in spatial order
#ifndef OBB_ORDER_MIN_BOXES
#define OBB_ORDER_MIN_BOXES 1024
#endif
#ifndef OBB_ORDER_MIN_MB
#define OBB_ORDER_MIN_MB 64
#endif
namespace obbv {
constexpr int64_t kOrderMinBoxes = OBB_ORDER_MIN_BOXES;
constexpr int64_t kOrderMinLatticeBytes = int64_t(OBB_ORDER_MIN_MB) << 20;
constexpr int kPrepThreads = 128;   // four lanes prepare a box (prep_box)
constexpr int kPrepBoxes = kPrepThreads / 4;
constexpr int kGrab = OBB_GRAB;   // tiles per work grab
}  // namespace obbv

namespace obbv {
namespace {

// ---------------------------------------------------------------- quantise

// A box that is not finite, has a negative half-extent or does not fit 63 bits
// becomes an empty one.
__device__ __forceinline__ obb_qbox quantize_box(const obb_box& B, const LatticeFrame* __restrict__ f, int32_t* err)
{
    const float* raw = reinterpret_cast<const float*>(&B);
    bool bad = false;
    for (int q = 0; q < 12; ++q) bad |= !isfinite(raw[q]);
    double R[9];
    for (int b = 0; b < 3; ++b) {
        R[b] = (double)B.axis0[b];
        R[3 + b] = (double)B.axis1[b];
    }
    R[6] = __dsub_rn(__dmul_rn(R[1], R[5]), __dmul_rn(R[2], R[4]));
    R[7] = __dsub_rn(__dmul_rn(R[2], R[3]), __dmul_rn(R[0], R[5]));
    R[8] = __dsub_rn(__dmul_rn(R[0], R[4]), __dmul_rn(R[1], R[3]));
    double d[3];
    for (int b = 0; b < 3; ++b) d[b] = __dsub_rn(__dsub_rn((double)B.c[b], f->lo[b]), 0.5 * f->h[b]);
    obb_qbox o;
    o.reserved = 0;
    for (int a = 0; a < 3; ++a) {
        bad |= !(B.half[a] >= 0.0f);
        const double half = (double)B.half[a];
        double m = __dmul_rn(R[3 * a], d[0]);
        for (int b = 1; b < 3; ++b) m = __dadd_rn(m, __dmul_rn(R[3 * a + b], d[b]));
        const double lo = __dmul_rn(__dsub_rn(m, half), f->s32), hi = __dmul_rn(__dadd_rn(m, half), f->s32);
        bad |= !(fabs(lo) < 4.0e18 && fabs(hi) < 4.0e18);   // whole numbers there: floor and ceil change nothing
        o.b[2 * a] = __double2ll_rd(lo);
        o.b[2 * a + 1] = __double2ll_ru(hi);
        for (int b = 0; b < 3; ++b) o.n[3 * a + b] = normal_entry(R[3 * a + b], f, b);
    }
    if (bad) {
        atomicOr(err, kErrArg);
        for (int q = 0; q < 9; ++q) o.n[q] = q % 4 == 0 ? 1 : 0;
        for (int a = 0; a < 3; ++a) {
            o.b[2 * a] = 0;
            o.b[2 * a + 1] = -1;   // empty
        }
    }
    return o;
}

__global__ void k_quantize(const obb_box* __restrict__ boxes, int64_t K, const LatticeFrame* __restrict__ f,
                           obb_qbox* __restrict__ out, int32_t* err)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k < K) out[k] = quantize_box(boxes[k], f, err);
}

// ------------------------------------------------------------------- prep

// A launch of at most kShortTileBoxes boxes cuts its tiles by the warps of the
// counting grid a box has (prep_box's warps), so that the grid is not left to
// a few warps walking full tiles (81 boxes at 360^3: 38.5 -> 31.8 us a call, 30
// at 1024^3: 87.5 -> 64.7; from 255 boxes on full tiles are as fast: 65.6
// against 68.8).
constexpr int32_t kShortTileBoxes = 128;

// Four lanes a box (prep_box), counts zeroed on the way; then the last
// block to finish (an atomic ticket, nothing waits) turns the tile counts into
// offsets: off[0..K] exclusive, off[K + 1] = 0 (the counting kernel's work
// counter).  kFloat: float boxes, quantised on the way (32,752 boxes at 1024^3:
// 29.6 us, 42 with a quantisation launch before it; three warps a block that
// share the FP64 work: 40 us).
template <bool kFloat>
__global__ void __launch_bounds__(kPrepThreads) k_prep(const obb_qbox* __restrict__ boxes,
                                                       const obb_box* __restrict__ fboxes,
                                                       const LatticeFrame* __restrict__ frame,
                                                       const int32_t* __restrict__ d_K, int32_t K_val,
                                                       const LatRef* __restrict__ lats, int32_t n_lats,
                                                       const int32_t* __restrict__ lat_of_box, const CountOpts o,
                                                       int32_t grid_warps, BoxPrep* __restrict__ prep,
                                                       int64_t* __restrict__ tiles,
                                                       int64_t* __restrict__ off,
                                                       unsigned long long* __restrict__ counts,
                                                       unsigned long long* __restrict__ points,
                                                       unsigned int* __restrict__ ticket,
                                                       uint32_t* __restrict__ bucket, unsigned int* __restrict__ hist,
                                                       int32_t scan_tiles, int32_t* err)
{
    static_assert(kPrepBoxes == 32, "a warp quantises the block's boxes");
    const int64_t k = blockIdx.x * (int64_t)kPrepBoxes + (threadIdx.x >> 2);
    const int32_t K = d_K ? *d_K : K_val;
    __shared__ obb_qbox sq[kFloat ? kPrepBoxes : 1];
    if (kFloat) {
        const int64_t f = blockIdx.x * (int64_t)kPrepBoxes + threadIdx.x;
        if (threadIdx.x < 32 && f < K) sq[threadIdx.x] = quantize_box(fboxes[f], frame, err);
        __syncthreads();
    }
    // warps of the counting grid per box, when there are few boxes
    const int32_t warps = K > 0 && K <= kShortTileBoxes ? grid_warps / K : 0;
    const bool on = k < K;
    int64_t nt = 0;
    if (__any_sync(0xffffffffu, on))
        nt = prep_box(!on ? nullptr : kFloat ? &sq[threadIdx.x >> 2] : boxes + k, on && lat_of_box ? lat_of_box[k] : 0,
                      lats, n_lats, o, warps, on ? &prep[k] : nullptr, err);
    __syncwarp();   // the box's preparation is its four lanes' work
    if (on && (threadIdx.x & 3) == 0) {
        counts[k] = 0;
        if (points) points[k] = 0;
        tiles[k] = nt;
        if (bucket) {
            // spatial order: the 16^3 Morton cell of the centre of the box's
            // index-space rectangle (clamped to the lattice)
            const BoxPrep& p = prep[k];
            const int32_t N = max(p.latN, 1);
            const int64_t c[3] = {(int64_t)p.i0 + p.span / 2, (int64_t)p.j0 + p.nj / 2, (int64_t)p.k0 + p.nk / 2};
            uint32_t key = 0;
            for (int a = 0; a < 3; ++a) {
                const uint32_t q = (uint32_t)min(max(c[a] * 16 / N, (int64_t)0), (int64_t)15);
                for (int bit = 0; bit < 4; ++bit) key |= ((q >> bit) & 1u) << (3 * bit + a);
            }
            if (n_lats > 1) {
                // several lattices: lattice-major, each lattice's share of the
                // buckets split by the top bits of the Morton cell
                int sub = 0;
                while (sub < 12 && (n_lats << (sub + 1)) <= kOrderBuckets) ++sub;
                key = (uint32_t)(((int64_t)p.lat * kOrderBuckets) / n_lats) + (key >> (12 - sub));
                key = min(key, (uint32_t)kOrderBuckets - 1);
            }
            bucket[k] = key;
            atomicAdd(&hist[key], 1u);
        }
    }
    // the last block's work: the spatial order's bucket starts, or (scan_tiles)
    // the tile offsets in the caller's order; otherwise the offsets come from
    // k_tile_sums / k_tile_offsets
    if (!bucket && !scan_tiles) return;
    // the block's writes, then one gpu-scope fence before its ticket
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
        if (last) __threadfence();
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    if (bucket) {
        // spatial order: the bucket counts become bucket starts (exclusive
        // scan, one warp, 128 buckets a lane); k_order_scatter,
        // k_tile_sums and k_tile_offsets follow
        const int lane = threadIdx.x & 31;
        constexpr int per = kOrderBuckets / 32;
        unsigned int run = 0;
        for (int q = 0; q < per; ++q) run += hist[lane * per + q];
        unsigned int x = run;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        unsigned int start = x - run;
        for (int q = 0; q < per; ++q) {
            const unsigned int v = hist[lane * per + q];
            hist[lane * per + q] = start;
            start += v;
        }
        if (threadIdx.x == 0) *ticket = 0;   // ready for the next launch
        return;
    }
    // exclusive scan of tiles[0..K) by the last block (one warp): chunks of
    // 8 x 32 consecutive values, a thread's eight in registers (eight loads in
    // flight), a warp scan of the thread sums, and a running carry
    const int lane = threadIdx.x & 31;
    int64_t carry = 0;
    for (int32_t base = 0; base < K; base += 256) {
        int64_t v[8];
        int64_t sum = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int32_t i = base + 8 * lane + q;
            v[q] = i < K ? tiles[i] : 0;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) sum += v[q];
        int64_t x = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        int64_t run = carry + x - sum;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int32_t i = base + 8 * lane + q;
            if (i < K) off[i] = run;
            run += v[q];
        }
        carry += __shfl_sync(0xffffffffu, x, 31);
    }
    if (threadIdx.x == 0) {
        off[K] = carry;
        off[K + 1] = 0;
        *ticket = 0;   // ready for the next launch
    }
}

// ---------------------------------------------------------- spatial order

// perm[start of the box's bucket + its place] = box, and the box's tile count
// at the same place (the place within a bucket depends on scheduling; counts
// do not depend on the order)
__global__ void k_order_scatter(const uint32_t* __restrict__ bucket, const int64_t* __restrict__ tiles,
                                const int32_t* __restrict__ d_K, int32_t K_val, unsigned int* __restrict__ hist,
                                int32_t* __restrict__ perm, int64_t* __restrict__ ptiles)
{
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t K = d_K ? *d_K : K_val;
    if (k >= K) return;
    const unsigned int pos = atomicAdd(&hist[bucket[k]], 1u);
    if (pos < (unsigned int)K) {
        perm[pos] = (int32_t)k;
        ptiles[pos] = tiles[k];
    }
}

// ---------------------------------------------------------- tile offsets

// Tile offsets in counting order (the boxes' own, or the spatial order's
// permuted copy), in two passes over blocks of 2,048
// positions (256 threads, 8 consecutive positions each): k_tile_sums writes
// each block's total; k_tile_offsets adds up the totals of the blocks before
// its own and scans its positions.  off[i] = tiles of the boxes at positions
// 0..i-1, off[K] = all tiles, off[K + 1] = 0 (the counting kernel's work
// counter).
constexpr int kScanPer = 8;
static_assert(256 * kScanPer == kScanBlock, "offset scan: 256 threads x kScanPer positions per block");

__global__ void __launch_bounds__(256) k_tile_sums(const int64_t* __restrict__ tiles,
                                                    const int32_t* __restrict__ d_K, int32_t K_val,
                                                    int64_t* __restrict__ bsum)
{
    __shared__ int64_t ws[8];
    const int32_t K = d_K ? *d_K : K_val;
    const int64_t base = (int64_t)blockIdx.x * kScanBlock + threadIdx.x * kScanPer;
    int64_t v = 0;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) v += base + q < K ? tiles[base + q] : 0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t t = 0;
        for (int w = 0; w < 8; ++w) t += ws[w];
        bsum[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(256) k_tile_offsets(const int64_t* __restrict__ tiles,
                                                       const int64_t* __restrict__ bsum,
                                                       const int32_t* __restrict__ d_K, int32_t K_val,
                                                       int64_t* __restrict__ off)
{
    __shared__ int64_t ws[8];
    __shared__ int64_t before;
    const int32_t K = d_K ? *d_K : K_val;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    // the totals of the blocks before this one
    int64_t p = 0;
    for (int32_t b = threadIdx.x; b < (int32_t)blockIdx.x; b += 256) p += bsum[b];
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    if (lane == 0) ws[w] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t t = 0;
        for (int i = 0; i < 8; ++i) t += ws[i];
        before = t;
    }
    __syncthreads();
    // this block's positions: a thread's eight in registers, then an exclusive
    // scan of the thread sums (warp shuffles, then across the 8 warps)
    const int64_t base = (int64_t)blockIdx.x * kScanBlock + threadIdx.x * kScanPer;
    int64_t v[kScanPer];
    int64_t sum = 0;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        v[q] = base + q < K ? tiles[base + q] : 0;
        sum += v[q];
    }
    int64_t x = sum;
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();   // ws is reused
    if (lane == 31) ws[w] = x;
    __syncthreads();
    int64_t wbefore = 0;
    for (int i = 0; i < w; ++i) wbefore += ws[i];
    int64_t run = before + wbefore + x - sum;
#pragma unroll
    for (int q = 0; q < kScanPer; ++q) {
        if (base + q < K) off[base + q] = run;
        run += v[q];
    }
    // positions past K hold 0, so the thread whose eight positions include K
    // ends with run = off[K] (the launch has K_cap / 2048 + 1 blocks, so it exists)
    if (base <= K && K < base + kScanPer) {
        off[K] = run;
        off[K + 1] = 0;
    }
}

// ------------------------------------------------------- batched requests

// off[r] = boxes of requests 0..r-1 (each request's count clamped to its
// capacity), off[n] and *d_total = all of them; one block of 1024 threads
__global__ void __launch_bounds__(1024) k_batch_offsets(const BatchReq* __restrict__ reqs, int32_t n,
                                                        int64_t* __restrict__ off, int32_t* __restrict__ d_total)
{
    __shared__ int64_t part[1024];
    const int t = threadIdx.x;
    const int32_t per = (n + 1023) / 1024;
    const int32_t b0 = min(n, t * per), b1 = min(n, b0 + per);
    int64_t sum = 0;
    for (int32_t r = b0; r < b1; ++r) sum += min((int64_t)max(*reqs[r].d_K, 0), reqs[r].cap);
    part[t] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int64_t v = t >= o ? part[t - o] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int64_t run = part[t] - sum;
    for (int32_t r = b0; r < b1; ++r) {
        off[r] = run;
        run += min((int64_t)max(*reqs[r].d_K, 0), reqs[r].cap);
    }
    if (t == 1023) {
        off[n] = part[1023];
        *d_total = (int32_t)part[1023];
    }
}

// the request of combined position j: the last r with off[r] <= j
__device__ __forceinline__ int32_t batch_request(const int64_t* __restrict__ off, int32_t n, int64_t j)
{
    int32_t lo = 0, hi = n;   // off[lo] <= j < off[hi]
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (off[mid] <= j) lo = mid;
        else hi = mid;
    }
    return lo;
}

__global__ void k_batch_gather(const BatchReq* __restrict__ reqs, int32_t n, const int64_t* __restrict__ off,
                               obb_qbox* __restrict__ boxes, int32_t* __restrict__ lat_of_box)
{
    const int64_t total = off[n];
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < total; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = batch_request(off, n, j);
        boxes[j] = reqs[r].boxes[j - off[r]];
        lat_of_box[j] = reqs[r].lat;
    }
}

__global__ void k_batch_scatter(const BatchReq* __restrict__ reqs, int32_t n, const int64_t* __restrict__ off,
                                const uint64_t* __restrict__ counts, const uint64_t* __restrict__ points)
{
    const int64_t total = off[n];
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < total; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = batch_request(off, n, j);
        const int64_t i = j - off[r];
        reqs[r].counts[i] = counts[j];
        if (reqs[r].points) reqs[r].points[i] = points[j];
    }
}

// ------------------------------------------------------------------- scan

// Exclusive scan of n = *d_n int32 values (n <= cap) into out[0..n]; one block.
// out[0..n] = exclusive scan of in[0..n) (n = *d_n), one block of 1,024
// threads: chunks of 4,096 consecutive values (four per thread), a scan of
// the warp sums, and a running carry.
__global__ void __launch_bounds__(1024) k_scan_i32(const int32_t* __restrict__ in, int32_t* __restrict__ out,
                                                  const int32_t* __restrict__ d_n)
{
    __shared__ int32_t ws[32];
    __shared__ int32_t chunk_total;
    const int32_t n = *d_n;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int32_t carry = 0;
    for (int32_t c = 0; c < n; c += 4096) {
        const int32_t b = c + 4 * threadIdx.x;
        int32_t v[4], sum = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = b + q < n ? in[b + q] : 0;
            sum += v[q];
        }
        int32_t x = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[w] = x;
        __syncthreads();
        if (w == 0) {
            const int32_t t = ws[lane];
            int32_t u = t;
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, u, o);
                if (lane >= o) u += y;
            }
            ws[lane] = u - t;   // warps before
            if (lane == 31) chunk_total = u;
        }
        __syncthreads();
        int32_t run = carry + ws[w] + x - sum;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (b + q < n) out[b + q] = run;
            run += v[q];
        }
        carry += chunk_total;
        __syncthreads();   // ws and chunk_total are rewritten by the next chunk
    }
    if (threadIdx.x == 0) out[n] = carry;
}

// ------------------------------------------------------------------ count

// kProf: the launch adds up its algorithmic bytes, rows and rank rows into
// acc[0], acc[1], acc[3]; every launch adds its in-domain points into *dom.
// kMinB: resident blocks per SM the register budget aims at.
template <bool kProf, int kMinB>
__global__ void __launch_bounds__(256, kMinB) k_count(const BoxPrep* __restrict__ prep,
                                               const int64_t* __restrict__ off,
                                               const int32_t* __restrict__ d_K, int32_t K_val,
                                               unsigned long long* __restrict__ counts,
                                               unsigned long long* __restrict__ points,
                                               unsigned long long* __restrict__ acc,
                                               unsigned long long* __restrict__ dom,
                                               const int32_t* __restrict__ perm)
{
    uint32_t my_bytes = 0, my_rows = 0, my_rank = 0, my_dom = 0;
    const int lane = threadIdx.x & 31;
    const int32_t K = d_K ? *d_K : K_val;
    const int64_t total = off[K];
    unsigned long long* next = reinterpret_cast<unsigned long long*>(const_cast<int64_t*>(off + K + 1));
    // warps take runs of kGrab consecutive tiles from a global counter; within a
    // run the box and the tile coordinates advance incrementally
    // b: position in the launch's order; bi: the box there (perm[b], or b)
    int64_t c = 0, c_end = 0, box_end = 0;
    int32_t b = 0, bi = 0, tj = 0, tk = 0, ntj = 1;
    for (;;) {
        if (c == c_end) {
            unsigned long long g = 0;
            if (lane == 0) g = atomicAdd(next, (unsigned long long)kGrab);
            c = (int64_t)__shfl_sync(0xffffffffu, g, 0);
            if (c >= total) break;
            c_end = min(c + (int64_t)kGrab, total);
            // the last box b with off[b] <= c: a 32-way search, one probe per lane
            int32_t lo = 0, hi = K;   // off[lo] <= c < off[hi]
            while (hi - lo > 1) {
                const int32_t st = (hi - lo + 31) >> 5;
                const int32_t idx = lo + lane * st;
                const unsigned m = __ballot_sync(0xffffffffu, idx < hi && off[idx] <= c);
                lo += (31 - __clz(m)) * st;
                hi = min(hi, lo + st);
            }
            b = lo;
            bi = perm ? perm[b] : b;
            box_end = off[b + 1];
            const int32_t u = (int32_t)(c - off[b]);
            ntj = prep[bi].ntj;
            tk = u / ntj;
            tj = u - tk * ntj;
        } else if (c >= box_end) {
            ++b;
            while (off[b + 1] <= c) ++b;   // skip boxes without tiles
            bi = perm ? perm[b] : b;
            box_end = off[b + 1];
            ntj = prep[bi].ntj;
            tj = tk = 0;
        }
        uint32_t empty = 0, inbox = 0;
        if (!count_tile<kProf>(prep[bi], tj, tk, empty, inbox, my_bytes, my_rows, my_rank, my_dom)) {
            if (++tj == ntj) {
                tj = 0;
                ++tk;
            }
            ++c;
            continue;
        }
        empty = __reduce_add_sync(0xffffffffu, empty);
        inbox = __reduce_add_sync(0xffffffffu, inbox);
        if (lane == 0) {
            if (empty) atomicAdd(&counts[bi], (unsigned long long)empty);
            if (points && inbox) atomicAdd(&points[bi], (unsigned long long)inbox);
        }
        if (++tj == ntj) {
            tj = 0;
            ++tk;
        }
        ++c;
    }
    // in-domain points of this launch (always), and with profiling its
    // algorithmic bytes, non-empty rows and rank rows: block sums, one atomic
    // each
    if (kProf || dom) {
        __shared__ unsigned long long sh[4];
        if (threadIdx.x < 4) sh[threadIdx.x] = 0;
        __syncthreads();
        unsigned long long v[4] = {my_bytes, my_rows, my_dom, my_rank};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (!kProf && i != 2) continue;
            for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
            if (lane == 0 && v[i]) atomicAdd(&sh[i], v[i]);
        }
        __syncthreads();
        if (kProf && threadIdx.x < 4 && threadIdx.x != 2 && acc && sh[threadIdx.x])
            atomicAdd(&acc[threadIdx.x], sh[threadIdx.x]);
        if (threadIdx.x == 2 && dom && sh[2]) atomicAdd(dom, sh[2]);
    }
}

// ------------------------------------------------------------- few boxes

// quantize_box's arithmetic for one box by one warp, an entry of n, a term of
// a slab's centre or a bound a lane: 17 FP64 instructions in a row instead of
// 75, of 64 cycles each.
__device__ __forceinline__ void quantize_warp(const obb_box& B, const LatticeFrame* __restrict__ f, obb_qbox* out,
                                              int32_t* err)
{
    const int lane = threadIdx.x & 31;
    const float* raw = reinterpret_cast<const float*>(&B);
    bool bad = lane < 12 && !isfinite(raw[lane < 12 ? lane : 0]);
    const int e = lane < 9 ? lane : 0, a = e / 3, b = e - 3 * a, b1 = b == 2 ? 0 : b + 1, b2 = b == 0 ? 2 : b - 1;
    double r = __dsub_rn(__dmul_rn((double)B.axis0[b1], (double)B.axis1[b2]),
                         __dmul_rn((double)B.axis0[b2], (double)B.axis1[b1]));
    if (a < 2) r = (double)(a == 0 ? B.axis0[b] : B.axis1[b]);
    const int32_t n = normal_entry(r, f, b);
    const double t = __dmul_rn(r, __dsub_rn(__dsub_rn((double)B.c[b], f->lo[b]), 0.5 * f->h[b]));
    // lanes 0-5: bound lane & 1 of slab lane / 2
    const int sl = lane < 6 ? lane >> 1 : 0;
    double m = __shfl_sync(0xffffffffu, t, 3 * sl);
    m = __dadd_rn(m, __shfl_sync(0xffffffffu, t, 3 * sl + 1));
    m = __dadd_rn(m, __shfl_sync(0xffffffffu, t, 3 * sl + 2));
    const float half = B.half[sl];
    bad |= !(half >= 0.0f);
    const double v = __dmul_rn(__dadd_rn(m, (double)((lane & 1) ? half : -half)), f->s32);
    bad |= !(fabs(v) < 4.0e18);
    int64_t bound = (lane & 1) ? __double2ll_ru(v) : __double2ll_rd(v);
    const bool any = __any_sync(0xffffffffu, bad);   // an empty box then, as quantize_box leaves it
    if (any) {
        if (lane == 0) atomicOr(err, kErrArg);
        bound = -(lane & 1);
    }
    if (lane < 9) out->n[lane] = any ? (lane % 4 == 0 ? 1 : 0) : n;
    if (lane < 6) out->b[lane] = bound;
    if (lane == 12) out->reserved = 0;
}

// A few boxes in one launch: a cluster of kFewCluster
// blocks per box prepares it and counts its tiles, dealt out over the
// cluster's warps.  Such a call is latency: of the general path's six launches
// (box count, quantisation, preparation, two for the tile offsets, counting)
// and of lanes that walk 32 rows one after another.  Five boxes on 64^3: 27 us
// of kernels and 37 a call that way, 10 and 12 this way.  No scratch, no zeroed
// outputs: the cluster's sums meet in distributed shared memory and its first
// block writes them.  Boxes are quantised ones, or float ones quantised on the
// way (frame given).

constexpr int kFewThreads = 256;

// The one-launch path takes at most kFewMaxBoxes boxes, or kFewMaxCap where how
// many of a cap there are is only known on the device (most calls use little of
// their cap): eight blocks a box are a wave of blocks for every 38 boxes, and
// from about 100 on two launches are as fast (16 boxes 10 against 16 us, 64 16
// against 19, 96 17 and 20, 128 23 and 18, 256 40 and 20, 400 55 and 24; 64^3).
// Lattices of at most kFewMaxLatticeBytes (256^3), boxes times lattice bytes at most kFewMaxWork: a
// cluster per box cannot share a large box out over the whole machine as the
// general path's tile queue does (31 boxes of a tree's top levels at 1024^3: 267
// against 106 us; 255 boxes at 544^3: 134 against 84 us; seven at 340^3: 60
// against 73 us).  Profiling with counters (mode 1) needs the general path's.
constexpr int64_t kFewMaxBoxes = 96, kFewMaxCap = 256;
constexpr int64_t kFewMaxLatticeBytes = int64_t(2) << 20;
constexpr int64_t kFewMaxWork = int64_t(64) << 20;
constexpr int kFewCluster = 8;   // blocks per box (4: 12.8, 8: 9.6 us for the 16 to 32 boxes of a flooding wave)

__global__ void __launch_bounds__(kFewThreads) k_count_few(const obb_qbox* __restrict__ boxes,
                                                           const obb_box* __restrict__ fboxes,
                                                           const LatticeFrame* __restrict__ frame,
                                                           const int32_t* __restrict__ d_K, int32_t K,
                                                           const LatRef* __restrict__ lats, int32_t n_lats,
                                                           const int32_t* __restrict__ lat_of_box, const CountOpts o,
                                                           unsigned long long* __restrict__ counts,
                                                           unsigned long long* __restrict__ points,
                                                           unsigned long long* __restrict__ dom, int32_t* err)
{
    __shared__ BoxPrep p;
    __shared__ obb_qbox q;
    __shared__ int64_t s_tiles;
    __shared__ unsigned long long sum[3];   // empty, all and in-domain points
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    if (d_K) K = *d_K;
    constexpr int C = kFewCluster;
    const int32_t k = blockIdx.x / C, rank = blockIdx.x % C;
    if (k >= K) return;   // the whole cluster
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kFewThreads / 32;
    if (tid < 3) sum[tid] = 0;
    if (warp == 0) {
        if (fboxes) {
            quantize_warp(fboxes[k], frame, &q, err);
            __syncwarp();
        }
        const int64_t nt = prep_box(lane >= 4 ? nullptr : fboxes ? &q : boxes + k, lat_of_box ? lat_of_box[k] : 0, lats,
                                    n_lats, o, kWarps * C, &p, err);
        if (lane == 0) s_tiles = nt;
    }
    __syncthreads();
    unsigned long long v[3] = {0, 0, 0};
    uint32_t nb = 0, nr = 0, nk = 0;
    for (int64_t t = warp * C + rank; t < s_tiles; t += kWarps * C) {
        const int32_t tk = (int32_t)(t / p.ntj), tj = (int32_t)(t - (int64_t)tk * p.ntj);
        uint32_t e = 0, in = 0, in_dom = 0;
        if (count_tile<false>(p, tj, tk, e, in, nb, nr, nk, in_dom)) {
            v[0] += e;
            v[1] += in;
            v[2] += in_dom;
        }
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        for (int s = 16; s > 0; s >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], s);
        if (lane == 0 && v[i]) atomicAdd(&sum[i], v[i]);
    }
    cluster.sync();
    if (rank == 0 && tid < 3) {
        unsigned long long t = 0;
        for (int g = 0; g < C; ++g) t += *cluster.map_shared_rank(&sum[tid], g);
        if (tid == 0) counts[k] = t;
        else if (tid == 1 && points) points[k] = t;
        else if (tid == 2 && dom && t) atomicAdd(dom, t);
    }
    cluster.sync();   // no block leaves while its sums are read
}

// ---------------------------------------------------------------- report

__global__ void k_report(const LatticeFrame* __restrict__ f, const double* __restrict__ frames,
                         const obb_qbox* __restrict__ q, int32_t K, obb_box* __restrict__ out)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double* R = frames + 9 * (int64_t)k;
    const double s = 4294967296.0 / f->hmax;
    double c[3] = {0, 0, 0};
    obb_box o;
    for (int a = 0; a < 3; ++a) {
        double base = 0.0;
        for (int b = 0; b < 3; ++b) base += R[3 * a + b] * (f->lo[b] + 0.5 * f->h[b]);
        double lo = (double)q[k].b[2 * a] / s + base;
        double hi = (double)q[k].b[2 * a + 1] / s + base;
        double mid = 0.5 * (lo + hi);
        for (int b = 0; b < 3; ++b) c[b] += R[3 * a + b] * mid;
        o.half[a] = (float)(0.5 * (hi - lo));
    }
    for (int b = 0; b < 3; ++b) {
        o.c[b] = (float)c[b];
        o.axis0[b] = (float)R[b];
        o.axis1[b] = (float)R[3 + b];
    }
    out[k] = o;
}

__global__ void k_set_i32(int32_t* dst, int32_t v)
{
    *dst = v;
}

}  // namespace

obb_status set_device_int(obb_ctx* ctx, int32_t* d_dst, int32_t value)
{
    k_set_i32<<<1, 1, 0, ctx->stream>>>(d_dst, value);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

void launch_scan_i32(obb_ctx* ctx, const int32_t* in, int32_t* out, const int32_t* d_n)
{
    k_scan_i32<<<1, 1024, 0, ctx->stream>>>(in, out, d_n);
    note_launch(ctx);
}

void launch_box_report(obb_ctx* ctx, const obb_lattice* lat, const double* d_frames, const obb_qbox* d_q, int32_t K,
                       obb_box* d_out)
{
    if (K > 0) {
        k_report<<<(K + 31) / 32, 32, 0, ctx->stream>>>(lat->d_frame, d_frames, d_q, K, d_out);
        note_launch(ctx);
    }
}

obb_status quantize_boxes(obb_ctx* ctx, const obb_lattice* lat, const obb_box* d_boxes, int64_t K,
                          obb_qbox* d_out)
{
    if (K <= 0) return OBB_OK;
    k_quantize<<<(unsigned)((K + 31) / 32), 32, 0, ctx->stream>>>(d_boxes, K, lat->d_frame, d_out, ctx->d_err);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

// The counting kernel as a persistent grid (every resident block of every
// SM), in the register budget for the lattices' size: 5 blocks per SM for
// lattices of at least kOrderMinLatticeBytes (DRAM-resident: more warps to
// cover the loads), 4 below (L2-resident: more registers per thread).
template <bool kProf, int kMinB>
static void launch_count_v(obb_ctx* ctx, cudaStream_t s, const BoxPrep* prep, const int64_t* off, const int32_t* d_K,
                           int32_t K, uint64_t* counts, uint64_t* points, unsigned long long* acc, unsigned long long* dom,
                           const int32_t* perm)
{
    static int blocks_per_sm = 0;
    if (blocks_per_sm == 0) {
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_count<kProf, kMinB>, 256, 0) != cudaSuccess ||
            nb < 1)
            nb = 1;
        blocks_per_sm = nb;
    }
    k_count<kProf, kMinB><<<blocks_per_sm * ctx->num_sms, 256, 0, s>>>(
        prep, off, d_K, K, reinterpret_cast<unsigned long long*>(counts), reinterpret_cast<unsigned long long*>(points),
        acc, dom, perm);
}

static void launch_count(obb_ctx* ctx, cudaStream_t s, bool prof, int64_t lattice_bytes, const BoxPrep* prep,
                         const int64_t* off, const int32_t* d_K, int32_t K, uint64_t* counts, uint64_t* points,
                         unsigned long long* acc, unsigned long long* dom, const int32_t* perm)
{
    constexpr int kLarge = OBB_COUNT_MINB, kSmall = OBB_COUNT_MINB_SMALL;
    const bool large = lattice_bytes >= kOrderMinLatticeBytes;
    if (prof) {
        if (large) launch_count_v<true, kLarge>(ctx, s, prep, off, d_K, K, counts, points, acc, dom, perm);
        else launch_count_v<true, kSmall>(ctx, s, prep, off, d_K, K, counts, points, acc, dom, perm);
    } else {
        if (large) launch_count_v<false, kLarge>(ctx, s, prep, off, d_K, K, counts, points, acc, dom, perm);
        else launch_count_v<false, kSmall>(ctx, s, prep, off, d_K, K, counts, points, acc, dom, perm);
    }
}

// The last block of the preparation scans the tile counts of at most this many
// boxes (one warp, 256 a step), which saves the two scan launches: 127 to 255
// boxes 80 -> 69 us a call, 2,047 147.5 -> 144.5.
constexpr int64_t kPrepScanBoxes = 4096;

// warps of the counting kernel's grid (four blocks of 256 threads on an SM)
static int32_t count_grid_warps(const obb_ctx* ctx) { return 32 * ctx->num_sms; }

static bool few_boxes(const obb_ctx* ctx, const int32_t* d_K, int64_t K_cap, int64_t lattice_bytes)
{
    return ctx->prof != 1 && K_cap <= (d_K ? kFewMaxCap : kFewMaxBoxes) && lattice_bytes <= kFewMaxLatticeBytes &&
           K_cap * lattice_bytes <= kFewMaxWork;
}

// The events around a counting launch (with profiling on): one before, one after.
static obb_status prof_event(obb_ctx* ctx, cudaEvent_t* e)
{
    if (!ctx->prof) return OBB_OK;
    OBB_CK(ctx, cudaEventCreate(e));
    OBB_CK(ctx, cudaEventRecord(*e, ctx->stream));
    return OBB_OK;
}

static obb_status launch_few(obb_ctx* ctx, const LatRef* d_lats, int32_t n_lats, const int32_t* d_lat_of_box,
                             const obb_qbox* d_boxes, const obb_box* d_fboxes, const LatticeFrame* d_frame,
                             const int32_t* d_K, int64_t K_cap, uint64_t* d_counts, uint64_t* d_points,
                             unsigned long long* dom)
{
    constexpr int C = kFewCluster;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(K_cap * C));
    cfg.blockDim = dim3(kFewThreads);
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    OBB_TRY(prof_event(ctx, &e0));
    OBB_CK(ctx, cudaLaunchKernelEx(&cfg, k_count_few, d_boxes, d_fboxes, d_frame, d_K, (int32_t)K_cap, d_lats, n_lats,
                                   d_lat_of_box, CountOpts{ctx->tile_k, ctx->count_axis, ctx->count_rank},
                                   reinterpret_cast<unsigned long long*>(d_counts),
                                   reinterpret_cast<unsigned long long*>(d_points), dom, ctx->d_err));
    note_launch(ctx);
    OBB_TRY(prof_event(ctx, &e1));
    if (ctx->prof) ctx->prof_ev.emplace_back(e0, e1);
    return OBB_OK;
}

obb_status count_float_boxes(obb_ctx* ctx, const obb_lattice* lat, const obb_box* d_boxes, int64_t K,
                             uint64_t* d_counts, uint64_t* d_points)
{
    if (few_boxes(ctx, nullptr, K, (int64_t)lat->n_words * 8))
        return launch_few(ctx, lat->d_ref, 1, nullptr, nullptr, d_boxes, lat->d_frame, nullptr, K, d_counts, d_points,
                          ctx->d_prof + 2);
    return count_boxes_multi(ctx, lat->d_ref, 1, nullptr, nullptr, nullptr, K, d_counts, d_points,
                             (int64_t)lat->n_words * 8, d_boxes, lat->d_frame);
}

obb_status count_known(obb_ctx* ctx, const obb_lattice* lat, const obb_qbox* d_boxes, int64_t K, uint64_t* d_counts,
                       uint64_t* d_points)
{
    if (few_boxes(ctx, nullptr, K, (int64_t)lat->n_words * 8))
        return launch_few(ctx, lat->d_ref, 1, nullptr, d_boxes, nullptr, nullptr, nullptr, K, d_counts, d_points,
                          ctx->d_prof + 2);
    return count_boxes_multi(ctx, lat->d_ref, 1, nullptr, d_boxes, nullptr, K, d_counts, d_points,
                             (int64_t)lat->n_words * 8);
}

obb_status count_boxes(obb_ctx* ctx, const obb_lattice* lat, const obb_qbox* d_boxes, const int32_t* d_K,
                       int64_t K_cap, uint64_t* d_counts, uint64_t* d_points)
{
    if (ctx->count_defer) {
        // a batched step counts every layer's requests together (count_flush)
        ctx->count_defer->push_back(CountReq{lat, d_boxes, d_K, K_cap, d_counts, d_points});
        return OBB_OK;
    }
    return count_boxes_multi(ctx, lat->d_ref, 1, nullptr, d_boxes, d_K, K_cap, d_counts, d_points,
                             (int64_t)lat->n_words * 8);
}

obb_status count_boxes_multi(obb_ctx* ctx, const LatRef* d_lats, int32_t n_lats, const int32_t* d_lat_of_box,
                             const obb_qbox* d_boxes, const int32_t* d_K, int64_t K_cap, uint64_t* d_counts,
                             uint64_t* d_points, int64_t lattice_bytes, const obb_box* d_fboxes,
                             const LatticeFrame* d_frame)
{
    cudaStream_t s = ctx->stream;
    if (K_cap <= 0) return OBB_OK;
    if (K_cap > (int64_t(1) << 30)) return fail(ctx, OBB_ERR_RANGE, "too many boxes in one call");
    if (few_boxes(ctx, d_K, K_cap, lattice_bytes))
        return launch_few(ctx, d_lats, n_lats, d_lat_of_box, d_boxes, d_fboxes, d_frame, d_K, K_cap, d_counts,
                          d_points, ctx->d_prof + 2);
    BoxPrep* prep;
    int64_t *tiles, *off;
    unsigned int* ticket = ctx->d_ticket;
    uint32_t* bucket = nullptr;
    int32_t* perm = nullptr;
    int64_t *ptiles = nullptr, *bsum = nullptr;
    if (ctx->count_scratch) {
        // fixed scratch of a step being captured into a graph: its addresses must not move
        const CountScratch& cs = *ctx->count_scratch;
        if (K_cap > cs.cap) return fail(ctx, OBB_ERR_STATE, "count scratch of a captured step too small");
        prep = cs.prep;
        tiles = cs.tiles;
        off = cs.tiles + cs.cap;
        bsum = cs.bsum;
    } else {
        const int64_t nb = K_cap / kScanBlock + 1;
        OBB_CK(ctx, ctx->prep.reserve(sizeof(BoxPrep) * K_cap, s));
        OBB_CK(ctx, ctx->chunk_off.reserve(sizeof(int64_t) * (2 * K_cap + 2 + nb), s));
        prep = ctx->prep.as<BoxPrep>();
        tiles = ctx->chunk_off.as<int64_t>();
        off = tiles + K_cap;
        bsum = off + K_cap + 2;
        if (ctx->count_order && K_cap >= kOrderMinBoxes && lattice_bytes >= kOrderMinLatticeBytes) {
            // large batches on lattices too large for L2 are counted in
            // spatial order (boxes of every size over one region together, so
            // the region's lattice words are reused from L2)
            OBB_CK(ctx, ctx->order.reserve((2 * sizeof(int32_t) + sizeof(int64_t)) * K_cap, s));
            ptiles = reinterpret_cast<int64_t*>(ctx->order.as<char>());
            bucket = reinterpret_cast<uint32_t*>(ptiles + K_cap);
            perm = reinterpret_cast<int32_t*>(bucket + K_cap);
            OBB_CK(ctx, cudaMemsetAsync(ctx->d_order_hist, 0, kOrderBuckets * sizeof(unsigned int), s));
        }
    }
    const bool scan = !perm && K_cap <= kPrepScanBoxes;
    // the preparation kernel also zeroes counts and points (accumulated with atomics)
    const auto run_prep = [&](auto kernel) {
        kernel<<<(unsigned)((K_cap + kPrepBoxes - 1) / kPrepBoxes), kPrepThreads, 0, s>>>(
            d_boxes, d_fboxes, d_frame, d_K, (int32_t)K_cap, d_lats, n_lats, d_lat_of_box,
            CountOpts{ctx->tile_k, ctx->count_axis, ctx->count_rank}, count_grid_warps(ctx), prep, tiles, off,
            reinterpret_cast<unsigned long long*>(d_counts), reinterpret_cast<unsigned long long*>(d_points), ticket,
            bucket, bucket ? ctx->d_order_hist : nullptr, scan ? 1 : 0, ctx->d_err);
    };
    if (d_fboxes) run_prep(k_prep<true>);
    else run_prep(k_prep<false>);
    note_launch(ctx);
    // tile offsets (unless the preparation's last block has scanned them): an exclusive scan of the tile counts in counting order
    // (the spatial order's permuted copy, else the boxes' own order)
    const int64_t* scan_in = tiles;
    if (perm) {
        k_order_scatter<<<(unsigned)((K_cap + 255) / 256), 256, 0, s>>>(bucket, tiles, d_K, (int32_t)K_cap,
                                                                        ctx->d_order_hist, perm, ptiles);
        note_launch(ctx);
        scan_in = ptiles;
    }
    if (!scan) {
        const unsigned nsb = (unsigned)(K_cap / kScanBlock + 1);
        k_tile_sums<<<nsb, 256, 0, s>>>(scan_in, d_K, (int32_t)K_cap, bsum);
        k_tile_offsets<<<nsb, 256, 0, s>>>(scan_in, bsum, d_K, (int32_t)K_cap, off);
        note_launch(ctx, 2);
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    OBB_TRY(prof_event(ctx, &e0));
    launch_count(ctx, s, ctx->prof == 1, lattice_bytes, prep, off, d_K, (int32_t)K_cap, d_counts, d_points,
                 ctx->prof == 1 ? ctx->d_prof : nullptr, ctx->d_prof + 2, perm);
    note_launch(ctx);
    OBB_TRY(prof_event(ctx, &e1));
    if (ctx->prof) ctx->prof_ev.emplace_back(e0, e1);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

obb_status count_flush(obb_ctx* ctx, const std::vector<CountReq>& reqs, DevBuf& tables, DevBuf& scratch)
{
    cudaStream_t s = ctx->stream;
    const int32_t n = (int32_t)reqs.size();
    if (n == 0) return OBB_OK;
    if (n > (1 << 20)) return fail(ctx, OBB_ERR_RANGE, "too many counting requests in one batch");
    // lattice table and request table (host), uploaded into `tables`
    std::vector<const obb_lattice*> lats;
    std::vector<BatchReq> hreq(n);
    int64_t cap = 0, lattice_bytes = 0;
    for (int32_t r = 0; r < n; ++r) {
        const CountReq& q = reqs[r];
        int32_t li = 0;
        while (li < (int32_t)lats.size() && lats[li] != q.lat) ++li;
        if (li == (int32_t)lats.size()) {
            lats.push_back(q.lat);
            lattice_bytes += (int64_t)q.lat->n_words * 8;
        }
        hreq[r] = BatchReq{q.boxes, q.d_K, q.counts, q.points, q.K_cap, li, 0};
        cap += q.K_cap;
    }
    if (cap > (int64_t(1) << 30)) return fail(ctx, OBB_ERR_RANGE, "too many boxes in one batch");
    const size_t req_bytes = (sizeof(BatchReq) * n + 255) / 256 * 256;
    const size_t lat_bytes = (sizeof(LatRef) * lats.size() + 255) / 256 * 256;
    OBB_CK(ctx, tables.reserve(req_bytes + lat_bytes, s));
    BatchReq* d_req = tables.as<BatchReq>();
    LatRef* d_lat = reinterpret_cast<LatRef*>(tables.as<char>() + req_bytes);
    std::vector<LatRef> hlat(lats.size());
    for (size_t i = 0; i < lats.size(); ++i) hlat[i] = lats[i]->ref;
    // pinned staging keeps the copies asynchronous (the tables are small)
    void* h = nullptr;
    OBB_CK(ctx, cudaMallocHost(&h, req_bytes + lat_bytes));
    memcpy(h, hreq.data(), sizeof(BatchReq) * n);
    memcpy(static_cast<char*>(h) + req_bytes, hlat.data(), sizeof(LatRef) * hlat.size());
    cudaError_t e = cudaMemcpyAsync(d_req, h, req_bytes + lat_bytes, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the staging is freed below
    cudaFreeHost(h);
    OBB_CK(ctx, e);
    // combined scratch: offsets [n + 1], total, boxes [cap], lattice of box [cap], counts and points [cap]
    const size_t off_b = (sizeof(int64_t) * (n + 1) + 255) / 256 * 256;
    const size_t box_b = (sizeof(obb_qbox) * cap + 255) / 256 * 256;
    const size_t li_b = (sizeof(int32_t) * cap + 255) / 256 * 256;
    const size_t cnt_b = (sizeof(uint64_t) * cap + 255) / 256 * 256;
    OBB_CK(ctx, scratch.reserve(off_b + 256 + box_b + li_b + 2 * cnt_b, s));
    char* b = scratch.as<char>();
    int64_t* off = reinterpret_cast<int64_t*>(b);
    int32_t* d_total = reinterpret_cast<int32_t*>(b + off_b);
    obb_qbox* boxes = reinterpret_cast<obb_qbox*>(b + off_b + 256);
    int32_t* lat_of_box = reinterpret_cast<int32_t*>(b + off_b + 256 + box_b);
    uint64_t* counts = reinterpret_cast<uint64_t*>(b + off_b + 256 + box_b + li_b);
    uint64_t* points = counts + cnt_b / sizeof(uint64_t);
    k_batch_offsets<<<1, 1024, 0, s>>>(d_req, n, off, d_total);
    const unsigned gb = (unsigned)std::min<int64_t>((cap + 255) / 256, 4 * (int64_t)ctx->num_sms);
    k_batch_gather<<<std::max(gb, 1u), 256, 0, s>>>(d_req, n, off, boxes, lat_of_box);
    note_launch(ctx, 2);
    OBB_TRY(count_boxes_multi(ctx, d_lat, (int32_t)lats.size(), lat_of_box, boxes, d_total, cap, counts, points,
                              lattice_bytes));
    k_batch_scatter<<<std::max(gb, 1u), 256, 0, s>>>(d_req, n, off, counts, points);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

}  // namespace obbv

// ---------------------------------------------------------------------------
// Outer volume without device allocation.
//
// Some callers cannot allocate device memory once they are running: a
// real-time collision or physics loop that works inside a fixed memory
// budget, or a host framework that owns the whole device memory pool and
// forbids allocations outside it.  This variant of the counting path takes
// its per-box scratch (count preparation, chunk counts and offsets, the box
// count) from one file-scope device array of fixed size instead of the
// context's growable buffers.  Every GPU that loads the library holds the
// array until the process exits.
// ---------------------------------------------------------------------------
namespace obbv {
namespace {

constexpr int64_t kNoAllocMaxBoxes = 4096;   // OBB_NOALLOC_MAX_BOXES in obbvar.h
constexpr size_t kNoAllocPrepBytes = sizeof(BoxPrep) * kNoAllocMaxBoxes;
constexpr size_t kNoAllocChunkBytes = sizeof(int64_t) * kNoAllocMaxBoxes;
constexpr size_t kNoAllocOffBytes = sizeof(int64_t) * (kNoAllocMaxBoxes + 2);
constexpr size_t kNoAllocOffsetChunks = (kNoAllocPrepBytes + 255) / 256 * 256;
constexpr size_t kNoAllocOffsetOff = kNoAllocOffsetChunks + (kNoAllocChunkBytes + 255) / 256 * 256;
constexpr size_t kNoAllocOffsetK = kNoAllocOffsetOff + (kNoAllocOffBytes + 255) / 256 * 256;
constexpr size_t kNoAllocBytes = kNoAllocOffsetK + 256;

// Shared by every call on a device; holds the last call's contents.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
unsigned char* g_noalloc_ptr[kNoAllocMaxDevices] = {};

// Device address of the array on `device` (looked up once per device, with
// that device current).  In host code the array's name is only a stand-in.
obb_status noalloc_scratch(obb_ctx* ctx, unsigned char** out)
{
    if (ctx->device < 0 || ctx->device >= kNoAllocMaxDevices) return fail(ctx, OBB_ERR_ARG, "device index too large");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[ctx->device]) {
        int prev = -1;
        OBB_CK(ctx, cudaGetDevice(&prev));
        if (prev != ctx->device) OBB_CK(ctx, cudaSetDevice(ctx->device));
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (prev != ctx->device) cudaSetDevice(prev);
        if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        g_noalloc_ptr[ctx->device] = static_cast<unsigned char*>(p);
    }
    *out = g_noalloc_ptr[ctx->device];
    return OBB_OK;
}

}  // namespace
}  // namespace obbv

extern "C" obb_status obb_outer_volume_q_noalloc(obb_ctx* ctx, const obb_lattice* lat, const obb_qbox* d_boxes,
                                                 int64_t K, uint64_t* d_counts, uint64_t* d_points)
{
    using namespace obbv;
    if (!ctx || !lat) return fail(ctx, OBB_ERR_ARG, "null argument");
    if (lat->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "lattice belongs to another context");
    if (K < 0) return fail(ctx, OBB_ERR_ARG, "negative K");
    if (K > kNoAllocMaxBoxes)
        return fail(ctx, OBB_ERR_RANGE,
                    "obb_outer_volume_q_noalloc takes at most " + std::to_string(kNoAllocMaxBoxes) +
                        " boxes per call (got " + std::to_string(K) + "); split the batch or use obb_outer_volume_q");
    if (K == 0) return OBB_OK;
    if (!d_boxes || !d_counts) return fail(ctx, OBB_ERR_ARG, "null argument");
    unsigned char* base = nullptr;
    OBB_TRY(noalloc_scratch(ctx, &base));
    BoxPrep* prep = reinterpret_cast<BoxPrep*>(base);
    int64_t* chunks = reinterpret_cast<int64_t*>(base + kNoAllocOffsetChunks);
    int64_t* off = reinterpret_cast<int64_t*>(base + kNoAllocOffsetOff);
    cudaStream_t s = ctx->stream;
    // the last 128 bytes of the count's slot hold the preparation blocks' ticket
    // (zero at load; every launch leaves it at zero again)
    unsigned int* ticket = reinterpret_cast<unsigned int*>(base + kNoAllocOffsetK + 128);
    // the preparation kernel also zeroes counts and points (accumulated with atomics)
    k_prep<false><<<(unsigned)((K + kPrepBoxes - 1) / kPrepBoxes), kPrepThreads, 0, s>>>(
        d_boxes, nullptr, nullptr, nullptr, (int32_t)K, lat->d_ref, 1, nullptr,
        CountOpts{ctx->tile_k, ctx->count_axis, ctx->count_rank}, count_grid_warps(ctx), prep, chunks, off,
        reinterpret_cast<unsigned long long*>(d_counts), reinterpret_cast<unsigned long long*>(d_points), ticket,
        nullptr, nullptr, 1, ctx->d_err);
    note_launch(ctx);
    launch_count(ctx, s, false, (int64_t)lat->n_words * 8, prep, off, nullptr, (int32_t)K, d_counts, d_points, nullptr,
                 nullptr, nullptr);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}
