// Patch division by flooding (Sec. 4.2.1 step 1), on the GPU.
//
// The boxes of a layer keep their frames and centres; the triangles are
// re-partitioned.  A triangle may only join a box of its group (the parent
// of its current cluster), so groups are independent and run side by side.
//   priority   per triangle: distance from its centroid (FP64, the mean of its
//              three float vertices) to the nearest centre of its group's
//              boxes, rounded to float, packed with the triangle index;
//   seeds      per group, its boxes in index order each take the nearest
//              untaken triangle of the group;
//   waves      a triangle is available once an edge neighbour of its group is
//              assigned (a group with none available falls back to its
//              unassigned triangle of smallest priority, with every box of the
//              group as candidate).  Exact mode takes the available triangle of
//              smallest priority per group per wave -- the paper's sequential
//              priority-queue order, since groups never interact -- and the
//              wavefront mode takes every available triangle at once.  A taken
//              triangle joins the candidate box (boxes holding one of its
//              neighbours) whose exact outer volume grows least (Eq. 12-13,
//              ties -> smaller box); in the wavefront mode several triangles
//              may join one box in a wave, each evaluated against the box as the
//              wave found it, and the box is recounted afterwards.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "counting.cuh"
#include "internal.h"

namespace obbv {
namespace {

constexpr int kMaxFloodCand = 8;   // boxes one triangle may choose between
constexpr int kFT = 128;

struct FloodRec {
    int32_t t, nk;
    int32_t k[kMaxFloodCand];
    int32_t e[kMaxFloodCand];   // eval slot of the grown box, -1 if unchanged
};

__device__ __forceinline__ unsigned long long tri_key(const float* __restrict__ V, const int32_t* __restrict__ F,
                                                      int32_t t, const double* c)
{
    double d2 = 0.0;
    for (int b = 0; b < 3; ++b) {
        double m = __dadd_rn((double)V[3 * (int64_t)F[3 * t] + b], (double)V[3 * (int64_t)F[3 * t + 1] + b]);
        m = __dadd_rn(m, (double)V[3 * (int64_t)F[3 * t + 2] + b]);
        m = __ddiv_rn(m, 3.0);
        const double d = __dsub_rn(m, c[b]);
        d2 = __dadd_rn(d2, __dmul_rn(d, d));
    }
    const float f = __double2float_rn(__dsqrt_rn(d2));
    return ((unsigned long long)__float_as_uint(f) << 32) | (unsigned long long)(uint32_t)t;
}

__device__ __forceinline__ void tri_proj(const int32_t* __restrict__ U, const int32_t* __restrict__ F, int32_t t,
                                         const int32_t* n, int64_t* e)
{
    for (int a = 0; a < 3; ++a) {
        e[2 * a] = INT64_MAX;
        e[2 * a + 1] = INT64_MIN;
    }
    for (int v = 0; v < 3; ++v) {
        const int32_t* P = U + 3 * (int64_t)F[3 * t + v];
        for (int a = 0; a < 3; ++a) {
            const int64_t d = (int64_t)n[3 * a] * P[0] + (int64_t)n[3 * a + 1] * P[1] + (int64_t)n[3 * a + 2] * P[2];
            e[2 * a] = min(e[2 * a], d);
            e[2 * a + 1] = max(e[2 * a + 1], d);
        }
    }
}

__global__ void k_fl_group(const int32_t* __restrict__ assign, const int32_t* __restrict__ parent, int64_t T,
                           int32_t* __restrict__ group, int32_t* __restrict__ nassign)
{
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= T) return;
    group[t] = parent[assign[t]];
    nassign[t] = -1;
}

__global__ void k_fl_box_count(const int32_t* __restrict__ parent, int32_t K, int32_t* __restrict__ gcount,
                               int32_t* err)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const int32_t g = parent[k];
    if (g < 0 || g >= K) {
        atomicOr(err, kErrArg);
        return;
    }
    atomicAdd(&gcount[g], 1);
}

__global__ void k_fl_box_fill(const int32_t* __restrict__ parent, int32_t K, const int32_t* __restrict__ gstart,
                              int32_t* __restrict__ gfill, int32_t* __restrict__ gbox)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const int32_t g = parent[k];
    gbox[gstart[g] + atomicAdd(&gfill[g], 1)] = k;
}

// ascending box order inside each group
__global__ void k_fl_box_sort(const int32_t* __restrict__ gstart, int32_t K, int32_t* __restrict__ gbox)
{
    int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= K) return;
    for (int32_t i = gstart[g] + 1; i < gstart[g + 1]; ++i)
        for (int32_t j = i; j > gstart[g] && gbox[j - 1] > gbox[j]; --j) {
            const int32_t x = gbox[j];
            gbox[j] = gbox[j - 1];
            gbox[j - 1] = x;
        }
}

__global__ void k_fl_keys(const float* __restrict__ V, const int32_t* __restrict__ F, int64_t T,
                          const int32_t* __restrict__ group, const int32_t* __restrict__ gstart,
                          const int32_t* __restrict__ gbox, const double* __restrict__ centre,
                          unsigned long long* __restrict__ key)
{
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= T) return;
    const int32_t g = group[t];
    unsigned long long best = ~0ull;
    for (int32_t i = gstart[g]; i < gstart[g + 1]; ++i) {
        const unsigned long long k = tri_key(V, F, (int32_t)t, centre + 3 * (int64_t)gbox[i]);
        best = k < best ? k : best;
    }
    key[t] = best;
}

// Seeds: one block per group; its boxes in index order take the nearest
// triangle of the group not taken by an earlier box.  The group's triangles
// are the members of the clusters whose parent is the group.
__global__ void __launch_bounds__(kFT) k_fl_seed(const float* __restrict__ V, const int32_t* __restrict__ F,
                                                 const int32_t* __restrict__ gstart, const int32_t* __restrict__ gbox,
                                                 const int32_t* __restrict__ members,
                                                 const int32_t* __restrict__ mstart,
                                                 const double* __restrict__ centre, int32_t* __restrict__ nassign,
                                                 int32_t* __restrict__ seed, int32_t* err)
{
    __shared__ unsigned long long red[kFT / 32];
    __shared__ int32_t taken[kMaxFloodCand];
    const int32_t g = blockIdx.x;
    const int32_t b0 = gstart[g], b1 = gstart[g + 1];
    if (b1 - b0 > kMaxFloodCand) {
        if (threadIdx.x == 0) atomicOr(err, kErrOverflow);
        return;
    }
    for (int32_t i = b0; i < b1; ++i) {
        const int32_t k = gbox[i];
        const double* c = centre + 3 * (int64_t)k;
        unsigned long long best = ~0ull;
        for (int32_t j = b0; j < b1; ++j) {
            const int32_t cl = gbox[j];   // the group's triangles: members of its old clusters
            for (int32_t m = mstart[cl] + threadIdx.x; m < mstart[cl + 1]; m += kFT) {
                const int32_t t = members[m];
                bool used = false;
                for (int32_t q = 0; q < i - b0; ++q) used |= taken[q] == t;
                if (used) continue;
                const unsigned long long kk = tri_key(V, F, t, c);
                best = kk < best ? kk : best;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long w = __shfl_xor_sync(0xffffffffu, best, o);
            best = w < best ? w : best;
        }
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long b = red[0];
            for (int w = 1; w < kFT / 32; ++w) b = red[w] < b ? red[w] : b;
            if (b == ~0ull) {
                atomicOr(err, kErrEmpty);
                taken[i - b0] = -1;
                seed[k] = -1;
            } else {
                const int32_t t = (int32_t)(b & 0xffffffffu);
                taken[i - b0] = t;
                seed[k] = t;
                nassign[t] = k;
            }
        }
        __syncthreads();
    }
}

// every box's slab from its seed triangle
__global__ void k_fl_seed_bounds(const int32_t* __restrict__ U, const int32_t* __restrict__ F,
                                 const int32_t* __restrict__ seed, int32_t K, obb_qbox* __restrict__ q)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const int32_t t = seed[k];
    if (t < 0) return;
    int64_t e[6];
    tri_proj(U, F, t, q[k].n, e);
    for (int i = 0; i < 6; ++i) q[k].b[i] = e[i];
}

__global__ void k_fl_reset(unsigned long long* __restrict__ gbest, unsigned long long* __restrict__ gfall,
                           int32_t K)
{
    int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= K) return;
    gbest[g] = ~0ull;
    gfall[g] = ~0ull;
}

__device__ __forceinline__ bool available(const int32_t* __restrict__ adj, const int32_t* __restrict__ group,
                                          const int32_t* __restrict__ nassign, int32_t t)
{
    bool a = false;
    for (int e = 0; e < 3; ++e) {
        const int32_t u = adj[3 * t + e];
        a |= nassign[u] >= 0 && group[u] == group[t];
    }
    return a;
}

// per group: smallest priority among available triangles (gbest) and among
// all unassigned ones (gfall)
__global__ void k_fl_minkeys(const int32_t* __restrict__ adj, const int32_t* __restrict__ group,
                             const int32_t* __restrict__ nassign, const unsigned long long* __restrict__ key,
                             int64_t T, unsigned long long* __restrict__ gbest, unsigned long long* __restrict__ gfall)
{
    int64_t tt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tt >= T) return;
    const int32_t t = (int32_t)tt;
    if (nassign[t] >= 0) return;
    const int32_t g = group[t];
    atomicMin(&gfall[g], key[t]);
    if (available(adj, group, nassign, t)) atomicMin(&gbest[g], key[t]);
}

__global__ void k_fl_select(const int32_t* __restrict__ U, const int32_t* __restrict__ F,
                            const int32_t* __restrict__ adj, const int32_t* __restrict__ group,
                            const int32_t* __restrict__ nassign, const unsigned long long* __restrict__ key,
                            int64_t T, const unsigned long long* __restrict__ gbest,
                            const unsigned long long* __restrict__ gfall, const int32_t* __restrict__ gstart,
                            const int32_t* __restrict__ gbox, const obb_qbox* __restrict__ q, int32_t wavefront,
                            FloodRec* __restrict__ rec, obb_qbox* __restrict__ evals, int32_t* __restrict__ ctr,
                            int32_t rec_cap, int32_t eval_cap, int32_t* err)
{
    int64_t tt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (tt >= T) return;
    const int32_t t = (int32_t)tt;
    if (nassign[t] >= 0) return;
    const int32_t g = group[t];
    const bool avail = available(adj, group, nassign, t);
    bool take;
    if (gbest[g] != ~0ull) take = wavefront ? avail : key[t] == gbest[g];
    else take = key[t] == gfall[g];
    if (!take) return;
    FloodRec r;
    r.t = t;
    r.nk = 0;
    if (avail) {
        for (int e = 0; e < 3; ++e) {
            const int32_t u = adj[3 * t + e];
            const int32_t k = nassign[u];
            if (k < 0 || group[u] != g) continue;
            bool dup = false;
            for (int i = 0; i < r.nk; ++i) dup |= r.k[i] == k;
            if (!dup) r.k[r.nk++] = k;
        }
    } else {
        const int32_t nb = gstart[g + 1] - gstart[g];
        if (nb > kMaxFloodCand) {
            atomicOr(err, kErrOverflow);
            return;
        }
        for (int i = 0; i < nb; ++i) r.k[r.nk++] = gbox[gstart[g] + i];
    }
    for (int i = 0; i < r.nk; ++i) {
        const obb_qbox& qk = q[r.k[i]];
        int64_t pr[6];
        tri_proj(U, F, t, qk.n, pr);
        obb_qbox gq = qk;
        bool grew = false;
        for (int a = 0; a < 3; ++a) {
            if (pr[2 * a] < gq.b[2 * a]) {
                gq.b[2 * a] = pr[2 * a];
                grew = true;
            }
            if (pr[2 * a + 1] > gq.b[2 * a + 1]) {
                gq.b[2 * a + 1] = pr[2 * a + 1];
                grew = true;
            }
        }
        r.e[i] = -1;
        if (grew) {
            const int32_t ei = atomicAdd(&ctr[1], 1);
            if (ei >= eval_cap) {
                atomicOr(err, kErrOverflow);
                return;
            }
            evals[ei] = gq;
            r.e[i] = ei;
        }
    }
    const int32_t ri = atomicAdd(&ctr[0], 1);
    if (ri >= rec_cap) {
        atomicOr(err, kErrOverflow);
        return;
    }
    rec[ri] = r;
}

// best box per taken triangle (smallest growth, ties -> smaller box) and, in
// exact mode, the box update (one taken triangle per group, so the boxes
// touched are distinct)
__global__ void k_fl_apply(const int32_t* __restrict__ U, const int32_t* __restrict__ F,
                           const FloodRec* __restrict__ rec, const int32_t* __restrict__ ctr,
                           const obb_qbox* __restrict__ evals, const uint64_t* __restrict__ ecount,
                           int32_t wavefront, int32_t* __restrict__ nassign, obb_qbox* __restrict__ q,
                           uint64_t* __restrict__ obv, uint8_t* __restrict__ changed, int32_t* __restrict__ left)
{
    int32_t ri = blockIdx.x * blockDim.x + threadIdx.x;
    if (ri >= ctr[0]) return;
    const FloodRec& r = rec[ri];
    int bi = -1;
    int64_t bc = 0;
    int32_t bk = INT32_MAX;
    for (int i = 0; i < r.nk; ++i) {
        const int32_t k = r.k[i];
        const int64_t c = r.e[i] >= 0 ? (int64_t)ecount[r.e[i]] - (int64_t)obv[k] : 0;
        if (bi < 0 || c < bc || (c == bc && k < bk)) {
            bi = i;
            bc = c;
            bk = k;
        }
    }
    nassign[r.t] = bk;
    atomicSub(left, 1);
    if (!wavefront) {
        if (r.e[bi] >= 0) {
            for (int i = 0; i < 6; ++i) q[bk].b[i] = evals[r.e[bi]].b[i];
            obv[bk] = ecount[r.e[bi]];
        }
    } else {
        int64_t pr[6];
        tri_proj(U, F, r.t, q[bk].n, pr);
        for (int a = 0; a < 3; ++a) {
            atomicMin(reinterpret_cast<long long*>(&q[bk].b[2 * a]), (long long)pr[2 * a]);
            atomicMax(reinterpret_cast<long long*>(&q[bk].b[2 * a + 1]), (long long)pr[2 * a + 1]);
        }
        changed[bk] = 1;
    }
}

__global__ void k_fl_compact(const uint8_t* __restrict__ changed, int32_t K, const obb_qbox* __restrict__ q,
                             obb_qbox* __restrict__ evals, int32_t* __restrict__ map, int32_t* __restrict__ n)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K || !changed[k]) return;
    const int32_t i = atomicAdd(n, 1);
    evals[i] = q[k];
    map[i] = k;
}

__global__ void k_fl_recount(const int32_t* __restrict__ map, const int32_t* __restrict__ n,
                             const uint64_t* __restrict__ cnt, uint64_t* __restrict__ obv,
                             uint8_t* __restrict__ changed)
{
    int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= *n) return;
    obv[map[i]] = cnt[i];
    changed[map[i]] = 0;
}

// world-space centres of the layer's boxes (the slab midpoints through the frame)
__global__ void k_fl_centres(const LatticeFrame* __restrict__ f, const double* __restrict__ frames,
                             const obb_qbox* __restrict__ q, int32_t K, double* __restrict__ out)
{
    int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= K) return;
    const double* R = frames + 9 * (int64_t)k;
    const double s = 4294967296.0 / f->hmax;
    double c[3] = {0.0, 0.0, 0.0};
    for (int a = 0; a < 3; ++a) {
        double base = 0.0;
        for (int b = 0; b < 3; ++b) base = __dadd_rn(base, __dmul_rn(R[3 * a + b], __dadd_rn(f->lo[b], 0.5 * f->h[b])));
        const double mid = __dadd_rn(__ddiv_rn(0.5 * ((double)q[k].b[2 * a] + (double)q[k].b[2 * a + 1]), s), base);
        for (int b = 0; b < 3; ++b) c[b] = __dadd_rn(c[b], __dmul_rn(R[3 * a + b], mid));
    }
    for (int b = 0; b < 3; ++b) out[3 * (int64_t)k + b] = c[b];
}

// ---- exact mode: every group on its own cluster
//
// A triangle's priority does not depend on the boxes and it becomes available
// once any neighbour of its group is assigned, so a group's whole order is
// fixed before any box is chosen (k_fl_order), and groups never interact: a
// cluster of blocks takes its group through that order (k_fl_run), counting
// the boxes that a triangle would grow on the way.  A wave per launch instead
// takes eight launches and two round trips to the host for one triangle of
// each group (10k triangles, 16 groups: 623 waves, 46.7 ms a call; this way 2.7 ms:
// 0.38 ms for the orders, 3.0 us a triangle after that, mostly the latency of
// preparing and counting one or two grown boxes).
//
// A group's triangles are numbered locally (base[g] + 0, 1, ..., by its old
// clusters), with their neighbours, vertices and assignment side by side, so
// that its cluster works out of L1 and L2.

struct FloodTotals {
    unsigned long long evals;
    int32_t groups, longest;   // groups that have triangles left; the most that any has after its seeds
};

// nonempty groups, and every group's number of triangles
__global__ void k_fl_sizes(const int32_t* __restrict__ gstart, const int32_t* __restrict__ gbox,
                           const int32_t* __restrict__ mstart, int32_t K, int32_t* __restrict__ gsize,
                           int32_t* __restrict__ glist, FloodTotals* __restrict__ tot)
{
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= K) return;
    int32_t n = 0;
    for (int32_t i = gstart[g]; i < gstart[g + 1]; ++i) n += mstart[gbox[i] + 1] - mstart[gbox[i]];
    gsize[g] = n;
    if (n > 0) {
        glist[atomicAdd(&tot->groups, 1)] = g;
        atomicMax(&tot->longest, n - (gstart[g + 1] - gstart[g]));
    }
}

// the groups whose order is not at its end (tot->groups zeroed before)
__global__ void k_fl_unfinished(const int32_t* __restrict__ gstart, const int32_t* __restrict__ base,
                                const int32_t* __restrict__ done, int32_t K, int32_t* __restrict__ glist,
                                FloodTotals* __restrict__ tot)
{
    const int32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < K && base[g + 1] - base[g] - (gstart[g + 1] - gstart[g]) > done[g])
        glist[atomicAdd(&tot->groups, 1)] = g;
}

// local numbers: block per group
__global__ void __launch_bounds__(kFT) k_fl_number(const int32_t* __restrict__ gstart, const int32_t* __restrict__ gbox,
                                                   const int32_t* __restrict__ members,
                                                   const int32_t* __restrict__ mstart,
                                                   const int32_t* __restrict__ base, int32_t* __restrict__ ltri,
                                                   int32_t* __restrict__ lid)
{
    const int32_t g = blockIdx.x;
    int32_t at = 0;
    for (int32_t i = gstart[g]; i < gstart[g + 1]; ++i) {
        const int32_t b0 = mstart[gbox[i]], n = mstart[gbox[i] + 1] - b0;
        for (int32_t m = threadIdx.x; m < n; m += kFT) {
            const int32_t t = members[b0 + m];
            ltri[base[g] + at + m] = t;
            lid[t] = at + m;
        }
        at += n;
    }
}

// per local triangle: neighbours of its group (local numbers, -1 = another
// group), snapped vertices, seed's box (its place among the group's boxes)
// or -1
__global__ void k_fl_local(const int32_t* __restrict__ U, const int32_t* __restrict__ F,
                           const int32_t* __restrict__ adj, int64_t T, const int32_t* __restrict__ ltri,
                           const int32_t* __restrict__ lid, const int32_t* __restrict__ group,
                           const int32_t* __restrict__ gstart, const int32_t* __restrict__ gbox,
                           const int32_t* __restrict__ nassign, int32_t* __restrict__ ladj,
                           int32_t* __restrict__ lvert, int8_t* __restrict__ lbox)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int32_t t = ltri[i], g = group[t];
    for (int e = 0; e < 3; ++e) {
        const int32_t u = adj[3 * (int64_t)t + e];
        ladj[3 * i + e] = group[u] == g ? lid[u] : -1;
        for (int c = 0; c < 3; ++c) lvert[9 * i + 3 * e + c] = U[3 * (int64_t)F[3 * (int64_t)t + e] + c];
    }
    int8_t s = -1;
    const int32_t k = nassign[t];
    for (int32_t b = gstart[g]; k >= 0 && b < gstart[g + 1]; ++b)
        if (gbox[b] == k) s = (int8_t)(b - gstart[g]);
    lbox[i] = s;
}

// triangles a launch takes from each group: 40 ms at 1024^3, a quarter of a second at worst (24,000 triangles in one
// group of two boxes that fill 2048^3)
constexpr int32_t kRunSteps = 4096;
// ... and the first launch of uneven groups (the longest more than twice the average) too many for eight blocks each,
// twice as many in every one after it: the blocks of groups that end sooner go to the others (24,000 triangles at
// 400^3, 125 groups of which the longest has 4,800: 615 -> 244 ms; groups of like size only wait for one another then,
// 10.1 -> 10.6 ms)
constexpr int32_t kRunFirst = 128;

// The order of a group's triangles after its seeds, a warp per group: the
// smallest priority among the available triangles (a list in the group's
// part of fkey / fid, state 1), else among all that are left; state 2 = taken.
// At most kRunSteps triangles a launch; prog[g] = {taken, listed} in between.
__global__ void __launch_bounds__(32) k_fl_order(const int32_t* __restrict__ glist, const int32_t* __restrict__ base,
                                                 const int32_t* __restrict__ gstart, const int32_t* __restrict__ ltri,
                                                 const unsigned long long* __restrict__ key, const int32_t* ladj,
                                                 const int8_t* lbox, uint8_t* state, unsigned long long* fkey,
                                                 int32_t* fid, int32_t* __restrict__ order,
                                                 int2* __restrict__ prog)
{
    const int32_t g = glist[blockIdx.x];
    const int64_t b0 = base[g];
    const int32_t n = base[g + 1] - base[g];
    const int lane = threadIdx.x;
    ladj += 3 * b0;
    lbox += b0;
    state += b0;
    fkey += b0;
    fid += b0;
    ltri += b0;
    order += b0;
    const int32_t first = prog[g].x, pops = n - (gstart[g + 1] - gstart[g]);
    int32_t F = prog[g].y;
    for (int32_t i = lane; first == 0 && i < n; i += 32) state[i] = lbox[i] >= 0 ? 2 : 0;
    __syncwarp();
    for (int32_t i = lane; first == 0 && i - lane < n; i += 32) {
        bool a = false;
        if (i < n && lbox[i] < 0)
            for (int e = 0; e < 3; ++e) {
                const int32_t u = ladj[3 * (int64_t)i + e];
                a |= u >= 0 && lbox[u] >= 0;
            }
        const unsigned m = __ballot_sync(0xffffffffu, a);
        if (a) {
            const int32_t p = F + __popc(m & ((1u << lane) - 1u));
            fkey[p] = key[ltri[i]];
            fid[p] = i;
            state[i] = 1;
        }
        F += __popc(m);
    }
    __syncwarp();
    const int32_t end = min(pops, first + kRunSteps);
    for (int32_t done = first; done < end; ++done) {
        unsigned long long best = ~0ull;
        int32_t at = -1;
        if (F > 0) {
            for (int32_t j = lane; j < F; j += 32)
                if (fkey[j] < best) {
                    best = fkey[j];
                    at = j;
                }
        } else {
            for (int32_t j = lane; j < n; j += 32)
                if (state[j] == 0 && key[ltri[j]] < best) {
                    best = key[ltri[j]];
                    at = j;
                }
        }
        // keys are distinct (they end with the triangle)
        const uint32_t hi = __reduce_min_sync(0xffffffffu, (uint32_t)(best >> 32));
        const uint32_t lo = __reduce_min_sync(0xffffffffu, (uint32_t)(best >> 32) == hi ? (uint32_t)best : ~0u);
        const int src = __ffs(__ballot_sync(0xffffffffu, at >= 0 && best == ((unsigned long long)hi << 32 | lo))) - 1;
        at = __shfl_sync(0xffffffffu, at, src);
        const int32_t i = F > 0 ? fid[at] : at;
        __syncwarp();
        if (F > 0) {
            --F;
            if (lane == 0) {
                fkey[at] = fkey[F];
                fid[at] = fid[F];
            }
        }
        if (lane == 0) {
            state[i] = 2;
            order[done] = i;
        }
        __syncwarp();
        // its neighbours that are neither taken nor listed
        const int32_t u = lane < 3 ? ladj[3 * (int64_t)i + lane] : -1;
        const unsigned same = __match_any_sync(0xffffffffu, u);
        const bool add = u >= 0 && lane == __ffs(same) - 1 && state[u] == 0;
        const unsigned m = __ballot_sync(0xffffffffu, add);
        if (add) {
            const int32_t p = F + __popc(m & ((1u << lane) - 1u));
            fkey[p] = key[ltri[u]];
            fid[p] = u;
            state[u] = 1;
        }
        F += __popc(m);
        __syncwarp();
    }
    if (lane == 0) prog[g] = make_int2(end, F);
}

constexpr int kRunThreads = 256;

struct FloodBox {
    int64_t b[6];
    unsigned long long obv;
    int32_t n[9];
};

// Groups through their orders: a cluster of C blocks per group.  The first
// warp of the cluster's first block walks the order; a triangle that lies
// inside its candidate boxes is assigned at once, and when it would grow some,
// the whole cluster prepares and counts the grown boxes (a warp prepares a box,
// the tiles are dealt out over the cluster's warps, the sums meet in the
// first block's shared memory) and the walker chooses.  done[g] triangles of
// the order are behind on entry, at most `steps` more on exit.
__global__ void __launch_bounds__(kRunThreads) k_fl_run(
    const int32_t* __restrict__ glist, const int32_t* __restrict__ base, const int32_t* __restrict__ gstart,
    const int32_t* __restrict__ gbox, const int32_t* __restrict__ order, const int32_t* __restrict__ ladj,
    const int32_t* __restrict__ lvert, int8_t* lbox, const LatRef* __restrict__ lats, const CountOpts o, int32_t C,
    int32_t steps, obb_qbox* __restrict__ q, uint64_t* __restrict__ obv, int32_t* __restrict__ done,
    unsigned long long* __restrict__ evals, unsigned long long* __restrict__ dom, int32_t* err)
{
    __shared__ BoxPrep prep[kMaxFloodCand];
    __shared__ obb_qbox ev[kMaxFloodCand];          // the grown boxes (the first block's are read by all)
    __shared__ int64_t tiles[kMaxFloodCand];
    __shared__ unsigned long long sum[kMaxFloodCand];
    __shared__ FloodBox box[kMaxFloodCand];
    __shared__ int32_t s_ne;
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int32_t g = glist[blockIdx.x / C], rank = blockIdx.x % C;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int kWarps = kRunThreads / 32;
    const int64_t b0 = base[g];
    const int32_t nb = gstart[g + 1] - gstart[g];   // at most kMaxFloodCand (k_fl_seed checked)
    const int32_t pops = base[g + 1] - base[g] - nb;
    const int32_t first = done[g], end = min(pops, first + steps);
    order += b0;
    ladj += 3 * b0;
    lvert += 9 * b0;
    lbox += b0;
    if (rank == 0 && tid < nb) {
        const int32_t k = gbox[gstart[g] + tid];
        for (int i = 0; i < 9; ++i) box[tid].n[i] = q[k].n[i];
        for (int i = 0; i < 6; ++i) box[tid].b[i] = q[k].b[i];
        box[tid].obv = obv[k];
    }
    __syncthreads();
    int32_t* ne_at = cluster.map_shared_rank(&s_ne, 0);
    const obb_qbox* ev_at = cluster.map_shared_rank(&ev[0], 0);
    unsigned long long* sum_at = cluster.map_shared_rank(&sum[0], 0);
    const bool walker = rank == 0 && warp == 0;
    int32_t step = first;
    int32_t i = 0, adj_next = -1, vert_next = 0, i_next = 0;
    auto fetch = [&](int32_t s) {   // the triangle of a step, its neighbours (lanes 0-2) and coordinates (lanes 0-8)
        if (s >= end) return;
        i_next = order[s];
        adj_next = lane < 3 ? ladj[3 * (int64_t)i_next + lane] : -1;
        vert_next = lane < 9 ? lvert[9 * (int64_t)i_next + lane] : 0;
    };
    unsigned cand = 0, grown = 0;   // candidate boxes and those that would grow (by place in the group)
    int64_t gb[6];                  // lane = box: its grown bounds
    unsigned long long n_evals = 0, n_dom = 0;
    if (walker) fetch(step);
    for (;;) {
        if (walker) {
            grown = 0;
            while (step < end && !grown) {
                i = i_next;
                const int32_t u = adj_next, vert = vert_next;
                fetch(step + 1);
                const int s = u >= 0 ? lbox[u] : -1;
                cand = __reduce_or_sync(0xffffffffu, s >= 0 ? 1u << s : 0u);
                if (!cand) cand = (1u << nb) - 1u;
                int32_t P[9];
#pragma unroll
                for (int c = 0; c < 9; ++c) P[c] = __shfl_sync(0xffffffffu, vert, c);
                bool grew = false;
                if (lane < kMaxFloodCand && (cand >> lane & 1u)) {
                    const FloodBox& B = box[lane];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        int64_t lo = B.b[2 * a], hi = B.b[2 * a + 1];
#pragma unroll
                        for (int v = 0; v < 3; ++v) {
                            const int64_t d = (int64_t)B.n[3 * a] * P[3 * v] + (int64_t)B.n[3 * a + 1] * P[3 * v + 1] +
                                              (int64_t)B.n[3 * a + 2] * P[3 * v + 2];
                            lo = min(lo, d);
                            hi = max(hi, d);
                        }
                        grew |= lo < B.b[2 * a] || hi > B.b[2 * a + 1];
                        gb[2 * a] = lo;
                        gb[2 * a + 1] = hi;
                    }
                }
                grown = __ballot_sync(0xffffffffu, grew);
                if (grown) {
                    if (grew) {
                        obb_qbox& E = ev[__popc(grown & ((1u << lane) - 1u))];
                        for (int c = 0; c < 9; ++c) E.n[c] = box[lane].n[c];
                        for (int c = 0; c < 6; ++c) E.b[c] = gb[c];
                        E.reserved = 0;
                    }
                    if (lane < kMaxFloodCand) sum[lane] = 0;
                } else {
                    // no candidate grows: equal (zero) growth, the smaller box
                    if (lane == 0) lbox[i] = (int8_t)(__ffs(cand) - 1);
                    __syncwarp();
                    ++step;
                }
            }
            if (lane == 0) s_ne = grown ? __popc(grown) : -1;
        }
        cluster.sync();
        const int ne = *ne_at;
        if (ne < 0) break;
        if (warp < ne) {
            const int64_t nt = prep_box(lane < 4 ? &ev_at[warp] : nullptr, 0, lats, 1, o, max(1, kWarps * C / ne),
                                        &prep[warp], err);
            if (lane == 0) tiles[warp] = nt;
        }
        __syncthreads();
        // the boxes' tiles one after another, dealt out over the cluster's warps
        int64_t t = warp * C + rank;
        for (int e = 0; e < ne; ++e) {
            uint32_t x0 = 0, x1 = 0, x2 = 0;
            unsigned long long empty = 0;
            for (; t < tiles[e]; t += kWarps * C) {
                const int32_t tk = (int32_t)(t / prep[e].ntj), tj = (int32_t)(t - (int64_t)tk * prep[e].ntj);
                uint32_t em = 0, in = 0, in_dom = 0;
                if (count_tile<false>(prep[e], tj, tk, em, in, x0, x1, x2, in_dom)) {
                    empty += em;
                    n_dom += in_dom;
                }
            }
            t -= tiles[e];
            for (int s = 16; s > 0; s >>= 1) empty += __shfl_xor_sync(0xffffffffu, empty, s);
            if (lane == 0 && empty) atomicAdd(&sum_at[e], empty);
        }
        cluster.sync();
        if (walker) {
            // the smallest growth of the outer volume, ties to the smaller box
            int64_t c = INT64_MAX;
            unsigned long long cnt = 0;
            const bool mine = lane < kMaxFloodCand && (cand >> lane & 1u);
            if (mine) {
                const bool grew = grown >> lane & 1u;
                if (grew) cnt = sum[__popc(grown & ((1u << lane) - 1u))];
                c = grew ? (int64_t)cnt - (int64_t)box[lane].obv : 0;
            }
            int64_t best = c;
            for (int s = 4; s > 0; s >>= 1) best = min(best, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)best, s));
            best = (int64_t)__shfl_sync(0xffffffffu, (long long)best, 0);
            const int win = __ffs(__ballot_sync(0xffffffffu, mine && c == best)) - 1;
            if (lane == win) {
                if (grown >> lane & 1u) {
                    for (int k = 0; k < 6; ++k) box[lane].b[k] = gb[k];
                    box[lane].obv = cnt;
                }
                lbox[i] = (int8_t)lane;
            }
            __syncwarp();
            n_evals += ne;
            ++step;
        }
    }
    if (rank == 0) {
        if (tid < nb) {
            const int32_t k = gbox[gstart[g] + tid];
            for (int c = 0; c < 6; ++c) q[k].b[c] = box[tid].b[c];
            obv[k] = box[tid].obv;
        }
        if (tid == 0) {
            done[g] = step;
            if (n_evals) atomicAdd(evals, n_evals);
        }
    }
    for (int s = 16; s > 0; s >>= 1) n_dom += __shfl_xor_sync(0xffffffffu, n_dom, s);
    if (lane == 0 && n_dom) atomicAdd(dom, n_dom);
    cluster.sync();   // no block leaves while the first one's shared memory is read
}

__global__ void k_fl_result(const int32_t* __restrict__ ltri, const int32_t* __restrict__ group,
                            const int32_t* __restrict__ gstart, const int32_t* __restrict__ gbox,
                            const int8_t* __restrict__ lbox, int64_t T, int32_t* __restrict__ assign)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int32_t t = ltri[i];
    assign[t] = gbox[gstart[group[t]] + lbox[i]];
}

struct FloodMem {
    obb_ctx* ctx = nullptr;
    std::vector<void*> ptrs;
    cudaError_t e = cudaSuccess;
    template <class T>
    T* get(size_t n)
    {
        void* p = nullptr;
        if (e == cudaSuccess) e = pool_alloc(&p, sizeof(T) * (n > 0 ? n : 1), ctx->stream);
        if (e == cudaSuccess) ptrs.push_back(p);
        return static_cast<T*>(p);
    }
    ~FloodMem()
    {
        for (void* p : ptrs) cudaFreeAsync(p, ctx->stream);
    }
};

// exact mode after the seeds: assignment into nassign, boxes and outer volumes into the layer
obb_status flood_exact(obb_ctx* ctx, obb_layer* L, FloodMem& mem, const int32_t* group, const int32_t* gstart,
                       const int32_t* gbox, const unsigned long long* key, int32_t* nassign, int32_t* waves,
                       int64_t* evals)
{
    cudaStream_t s = ctx->stream;
    const obb_lattice* lat = L->lat;
    const obb_mesh* mesh = lat->mesh;
    const int32_t K = L->K;
    const int64_t T = L->T;
    int32_t* gsize = mem.get<int32_t>(K);
    int32_t* base = mem.get<int32_t>((size_t)K + 1);
    int32_t* glist = mem.get<int32_t>(K);
    int32_t* done = mem.get<int32_t>(K);
    int2* prog = mem.get<int2>(K);
    int32_t* ltri = mem.get<int32_t>(T);
    int32_t* lid = mem.get<int32_t>(T);
    int32_t* ladj = mem.get<int32_t>(3 * (size_t)T);
    int32_t* lvert = mem.get<int32_t>(9 * (size_t)T);
    int32_t* order = mem.get<int32_t>(T);
    int32_t* fid = mem.get<int32_t>(T);
    unsigned long long* fkey = mem.get<unsigned long long>(T);
    int8_t* lbox = mem.get<int8_t>(T);
    uint8_t* state = mem.get<uint8_t>(T);
    FloodTotals* tot = mem.get<FloodTotals>(1);
    if (mem.e != cudaSuccess) return cuda_fail(ctx, mem.e, "flood scratch");
    const unsigned gT = (unsigned)((T + 255) / 256), gK = (unsigned)((K + 127) / 128);
    OBB_CK(ctx, cudaMemsetAsync(tot, 0, sizeof(FloodTotals), s));
    OBB_CK(ctx, cudaMemsetAsync(done, 0, sizeof(int32_t) * K, s));
    OBB_CK(ctx, cudaMemsetAsync(prog, 0, sizeof(int2) * K, s));
    k_fl_sizes<<<gK, 128, 0, s>>>(gstart, gbox, L->d_start, K, gsize, glist, tot);
    launch_scan_i32(ctx, gsize, base, layer_dev_K(L));
    k_fl_number<<<K, kFT, 0, s>>>(gstart, gbox, L->d_members, L->d_start, base, ltri, lid);
    k_fl_local<<<gT, 256, 0, s>>>(lat->d_fixed, mesh->d_tris, mesh->d_adj, T, ltri, lid, group, gstart, gbox, nassign,
                                  ladj, lvert, lbox);
    note_launch(ctx, 3);
    FloodTotals* h = reinterpret_cast<FloodTotals*>(host_stats(ctx));
    auto read = [&]() -> obb_status {
        OBB_CK(ctx, cudaMemcpyAsync(h, tot, sizeof(FloodTotals), cudaMemcpyDeviceToHost, s));
        return check_device_error(ctx);
    };
    OBB_TRY(read());
    if (h->groups <= 0) return fail(ctx, OBB_ERR_STATE, "a layer without groups");
    const int32_t longest = h->longest;
    const bool uneven = (int64_t)longest * h->groups > 2 * (T - K);
    for (int32_t taken = 0; taken < longest; taken += kRunSteps) {
        k_fl_order<<<h->groups, 32, 0, s>>>(glist, base, gstart, ltri, key, ladj, lbox, state, fkey, fid, order, prog);
        note_launch(ctx);
    }
    OBB_CK(ctx, cudaGetLastError());
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kRunThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const CountOpts o{ctx->tile_k, ctx->count_axis, ctx->count_rank};
    int32_t last = 0, steps = kRunSteps;
    for (int32_t taken = 0; taken < longest;) {
        // blocks per group: as many as keep every group's cluster on the chip (two blocks an SM)
        int32_t C = 8;
        while (C > 1 && (int64_t)C * h->groups > 2 * ctx->num_sms) C >>= 1;
        steps = C == 8 || !uneven ? kRunSteps : C != last ? kRunFirst : std::min(2 * steps, kRunSteps);
        last = C;
        cfg.gridDim = dim3((unsigned)h->groups * C);
        at[0].val.clusterDim.x = C;
        OBB_CK(ctx, cudaLaunchKernelEx(&cfg, k_fl_run, (const int32_t*)glist, (const int32_t*)base, gstart, gbox,
                                       (const int32_t*)order, (const int32_t*)ladj, (const int32_t*)lvert, lbox,
                                       (const LatRef*)lat->d_ref, o, C, steps, L->d_q, L->d_obv, done, &tot->evals,
                                       ctx->d_prof + 2, ctx->d_err));
        note_launch(ctx);
        taken += steps;   // by every group that is not at its end
        if (taken < longest) {
            OBB_CK(ctx, cudaMemsetAsync(&tot->groups, 0, sizeof(int32_t), s));
            k_fl_unfinished<<<gK, 128, 0, s>>>(gstart, base, done, K, glist, tot);
            note_launch(ctx);
        }
        OBB_TRY(read());
    }
    // a wave takes one triangle of every group that has any left: as many waves as the longest order has triangles
    *evals = (int64_t)h->evals;
    *waves = longest;
    k_fl_result<<<gT, 256, 0, s>>>(ltri, group, gstart, gbox, lbox, T, nassign);
    note_launch(ctx);
    return OBB_OK;
}

}  // namespace

obb_status flood_partition(obb_ctx* ctx, obb_layer* L, const double* d_centres, int32_t mode, obb_flood_stats* out)
{
    cudaStream_t s = ctx->stream;
    const obb_lattice* lat = L->lat;
    const obb_mesh* mesh = lat->mesh;
    const int32_t K = L->K;
    const int64_t T = L->T;
    if (mode != 0 && mode != 1) return fail(ctx, OBB_ERR_ARG, "flood mode must be 0 (exact) or 1 (wavefront)");
    OBB_TRY(layer_members(ctx, L));
    // With profiling counters (mode 1) the counting kernel's own launches, a wave at a time; and where the boxes are large
    // for the number of triangles: a group's cluster counts them with eight blocks, a wave with all of the machine.  A
    // run's counts grow with the boxes that grow (about the root of the triangles) and with N^3 of the points they
    // hold, the waves with the triangles: N^3 <= 6 10^7 sqrt(T).  Run against waves, ms: 144 triangles 2.6 : 4.7 at 512^3,
    // 10.4 : 5.4 at 1024^3; 1,920 triangles 50 : 113 at 1024^3, 122 : 116 at 1448^3, 282 : 121 at 2048^3; 24,000 at 2048^3
    // 1,296 : 1,583.
    const double side = (double)lat->frame.N;
    const bool run = mode == 0 && ctx->prof != 1 && side * side * side <= 6e7 * std::sqrt((double)T);
    FloodMem mem;
    mem.ctx = ctx;
    // exact mode takes at most one triangle per group and wave; the wavefront
    // up to every triangle, with three candidates unless it is a group's
    // fallback (up to kMaxFloodCand, at most one per group)
    const int32_t rec_cap = mode == 0 ? K : (int32_t)T;
    const int32_t eval_cap = (mode == 0 ? 0 : 3 * (int32_t)T) + kMaxFloodCand * K;
    int32_t* group = mem.get<int32_t>(T);
    int32_t* nassign = mem.get<int32_t>(T);
    unsigned long long* key = mem.get<unsigned long long>(T);
    int32_t* gcount = mem.get<int32_t>(K);
    int32_t* gstart = mem.get<int32_t>((size_t)K + 1);
    int32_t* gfill = mem.get<int32_t>(K);
    int32_t* gbox = mem.get<int32_t>(K);
    int32_t* seed = mem.get<int32_t>(K);
    double* centre = mem.get<double>(3 * (size_t)K);
    int32_t* ctr = mem.get<int32_t>(4);   // records, evals, unassigned, recount size
    // the waves' own
    unsigned long long *gbest = nullptr, *gfall = nullptr;
    FloodRec* rec = nullptr;
    obb_qbox* evals = nullptr;
    uint64_t* ecount = nullptr;
    uint8_t* changed = nullptr;
    int32_t* map = nullptr;
    if (!run) {
        gbest = mem.get<unsigned long long>(K);
        gfall = mem.get<unsigned long long>(K);
        rec = mem.get<FloodRec>(rec_cap);
        evals = mem.get<obb_qbox>(eval_cap);
        ecount = mem.get<uint64_t>(eval_cap);
        changed = mem.get<uint8_t>(K);
        map = mem.get<int32_t>(K);
    }
    if (mem.e != cudaSuccess) return cuda_fail(ctx, mem.e, "flood scratch");
    const unsigned gT = (unsigned)((T + 255) / 256), gK = (unsigned)((K + 127) / 128);
    if (d_centres) OBB_CK(ctx, cudaMemcpyAsync(centre, d_centres, sizeof(double) * 3 * K, cudaMemcpyDefault, s));
    else {
        k_fl_centres<<<gK, 128, 0, s>>>(lat->d_frame, L->d_frames, L->d_q, K, centre);
        note_launch(ctx);
    }
    k_fl_group<<<gT, 256, 0, s>>>(L->d_assign, L->d_parent, T, group, nassign);
    OBB_CK(ctx, cudaMemsetAsync(gcount, 0, sizeof(int32_t) * K, s));
    OBB_CK(ctx, cudaMemsetAsync(gfill, 0, sizeof(int32_t) * K, s));
    if (!run) OBB_CK(ctx, cudaMemsetAsync(changed, 0, K, s));
    k_fl_box_count<<<gK, 128, 0, s>>>(L->d_parent, K, gcount, ctx->d_err);
    note_launch(ctx, 2);
    OBB_TRY(set_device_int(ctx, ctr + 3, K));
    launch_scan_i32(ctx, gcount, gstart, ctr + 3);
    k_fl_box_fill<<<gK, 128, 0, s>>>(L->d_parent, K, gstart, gfill, gbox);
    k_fl_box_sort<<<gK, 128, 0, s>>>(gstart, K, gbox);
    k_fl_keys<<<gT, 256, 0, s>>>(mesh->d_verts, mesh->d_tris, T, group, gstart, gbox, centre, key);
    note_launch(ctx, 4);
    OBB_TRY(check_device_error(ctx));
    // seeds: the groups are the parents; L->d_start / d_members list the old clusters
    k_fl_seed<<<K, kFT, 0, s>>>(mesh->d_verts, mesh->d_tris, gstart, gbox, L->d_members, L->d_start, centre, nassign,
                                 seed, ctx->d_err);
    k_fl_seed_bounds<<<gK, 128, 0, s>>>(lat->d_fixed, mesh->d_tris, seed, K, L->d_q);
    note_launch(ctx, 2);
    OBB_TRY(check_device_error(ctx));
    OBB_TRY(count_known(ctx, lat, L->d_q, K, L->d_obv, nullptr));
    int64_t* h = host_stats(ctx);
    int32_t* hi = reinterpret_cast<int32_t*>(h);
    OBB_TRY(set_device_int(ctx, ctr + 2, (int32_t)(T - K)));
    obb_flood_stats st{};
    int64_t evals_total = 0;
    if (run) OBB_TRY(flood_exact(ctx, L, mem, group, gstart, gbox, key, nassign, &st.waves, &evals_total));
    while (!run) {
        OBB_CK(ctx, cudaMemcpyAsync(hi, ctr + 2, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        OBB_TRY(check_device_error(ctx));
        if (hi[0] <= 0) break;
        k_fl_reset<<<gK, 128, 0, s>>>(gbest, gfall, K);
        k_fl_minkeys<<<gT, 256, 0, s>>>(mesh->d_adj, group, nassign, key, T, gbest, gfall);
        OBB_CK(ctx, cudaMemsetAsync(ctr, 0, sizeof(int32_t) * 2, s));
        k_fl_select<<<gT, 256, 0, s>>>(lat->d_fixed, mesh->d_tris, mesh->d_adj, group, nassign, key, T, gbest, gfall,
                                       gstart, gbox, L->d_q, mode, rec, evals, ctr, rec_cap, eval_cap, ctx->d_err);
        note_launch(ctx, 3);
        OBB_TRY(count_boxes(ctx, lat, evals, ctr + 1, eval_cap, ecount, nullptr));
        k_fl_apply<<<(unsigned)((rec_cap + 127) / 128), 128, 0, s>>>(lat->d_fixed, mesh->d_tris, rec, ctr, evals,
                                                                     ecount, mode, nassign, L->d_q, L->d_obv,
                                                                     changed, ctr + 2);
        note_launch(ctx);
        if (mode == 1) {
            OBB_CK(ctx, cudaMemsetAsync(ctr + 3, 0, sizeof(int32_t), s));
            k_fl_compact<<<gK, 128, 0, s>>>(changed, K, L->d_q, evals, map, ctr + 3);
            note_launch(ctx);
            OBB_TRY(count_boxes(ctx, lat, evals, ctr + 3, K, ecount, nullptr));
            k_fl_recount<<<gK, 128, 0, s>>>(map, ctr + 3, ecount, L->d_obv, changed);
            note_launch(ctx);
        }
        OBB_CK(ctx, cudaMemcpyAsync(hi + 1, ctr + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        OBB_CK(ctx, cudaGetLastError());
        ++st.waves;
        OBB_CK(ctx, cudaStreamSynchronize(s));
        evals_total += hi[1];
    }
    OBB_CK(ctx, cudaMemcpyAsync(L->d_assign, nassign, sizeof(int32_t) * T, cudaMemcpyDeviceToDevice, s));
    layer_members_changed(L);
    OBB_CK(ctx, cudaMemsetAsync(layer_dirty(L), 1, K, s));
    OBB_CK(ctx, cudaMemsetAsync(layer_level(L), 0, sizeof(int32_t) * K, s));
    OBB_TRY(layer_members(ctx, L));
    OBB_TRY(check_device_error(ctx));
    st.box_evals = evals_total;
    if (out) *out = st;
    return OBB_OK;
}

}  // namespace obbv
