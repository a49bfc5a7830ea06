// Top-down construction of the binary OBB tree (Sec. 4.2.2) and its Eq. 7 score.
//
// Each level splits every node at the median of its triangles along the
// node's major axis and then runs Lloyd iterations restricted to siblings.
// The split is exact: key(t) = n_0 . (U_p + U_q + U_r) in int64 (three times
// the fixed-point centroid projected on the quantised major axis), ordered by
// (cluster, key, triangle); the first ceil(size / 2) triangles of a cluster go
// to child 2c, the rest to 2c + 1.  Clusters a block can walk select their
// median (k_split); larger ones are sorted with two stable radix sorts.
#include <cub/cub.cuh>

#include "internal.h"

namespace obbv {
namespace {

// n . (U_p + U_q + U_r) of triangle t
__device__ __forceinline__ int64_t split_key(const int32_t* __restrict__ U, const int32_t* __restrict__ F, int64_t t,
                                             const int32_t* n)
{
    int64_t s[3] = {0, 0, 0};
    for (int v = 0; v < 3; ++v) {
        const int32_t* P = U + 3 * (int64_t)F[3 * t + v];
        for (int b = 0; b < 3; ++b) s[b] += P[b];
    }
    return (int64_t)n[0] * s[0] + (int64_t)n[1] * s[1] + (int64_t)n[2] * s[2];
}

__global__ void k_split_keys(const int32_t* __restrict__ U, const int32_t* __restrict__ F, int64_t T,
                             const int32_t* __restrict__ assign, const obb_qbox* __restrict__ q,
                             int64_t* __restrict__ keys, int32_t* __restrict__ iota)
{
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= T) return;
    keys[t] = split_key(U, F, t, q[assign[t]].n);
    iota[t] = (int32_t)t;
}

constexpr int kSplitRank = 256;   // candidates ranked by comparing all with all

// Block per cluster: the median by (key, triangle), then every member's child.
// The order statistic is found by radix selection from the top significant bit
// of key - min key (then of the member's position, which ascends with the
// triangle), eight bits a pass, until at most kSplitRank candidates share the
// prefix; those are ranked against each other.  One pass is the rule.  The keys
// stay in L2 between passes; each thread reads back the ones it wrote.  Bound by
// the latency of the vertex gathers and of the block's barriers: a split of
// 10,000 triangles in 16 clusters takes 24 us as seen by the caller, of which
// 14 are its copy and synchronisation; the sorts' 22 launches took 152.
template <int NT>
__global__ void __launch_bounds__(NT) k_split(const int32_t* __restrict__ U, const int32_t* __restrict__ F,
                                              const int32_t* __restrict__ members, const int32_t* __restrict__ start,
                                              const obb_qbox* __restrict__ q, int64_t* keys,
                                              int32_t* __restrict__ child, int32_t* err)
{
    static_assert(NT >= 256, "a thread per bin");
    __shared__ int64_t s_lo[NT / 32], s_hi[NT / 32];
    __shared__ int32_t hist[256], wsum[8];
    __shared__ int32_t s_bin, s_need, s_cnt, s_fill;
    __shared__ uint64_t cw[kSplitRank], s_w;
    __shared__ int32_t cp[kSplitRank], s_p;
    const int32_t c = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t b0 = start[c], n = start[c + 1] - b0;
    if (n < 2) {
        if (tid == 0) {
            atomicOr(err, kErrEmpty);
            if (n == 1) child[members[b0]] = 2 * c;
        }
        return;
    }
    members += b0;
    keys += b0;
    const int32_t nn[3] = {q[c].n[0], q[c].n[1], q[c].n[2]};
    int64_t lo = INT64_MAX, hi = INT64_MIN;
    for (int32_t i = tid; i < n; i += NT) {
        const int64_t k = split_key(U, F, members[i], nn);
        keys[i] = k;
        lo = min(lo, k);
        hi = max(hi, k);
    }
    for (int d = 16; d > 0; d >>= 1) {
        lo = min(lo, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)lo, d));
        hi = max(hi, (int64_t)__shfl_xor_sync(0xffffffffu, (long long)hi, d));
    }
    if (lane == 0) {
        s_lo[warp] = lo;
        s_hi[warp] = hi;
    }
    __syncthreads();
    for (int w = 0; w < NT / 32; ++w) {
        lo = min(lo, s_lo[w]);
        hi = max(hi, s_hi[w]);
    }
    const uint64_t range = (uint64_t)hi - (uint64_t)lo;
    int kb = range ? 64 - __clzll((long long)range) : 0;   // key bits and position bits not yet fixed
    int pb = 32 - __clz(n - 1);
    uint64_t kv = 0;                                       // those fixed
    int32_t pv = 0;
    int32_t need = (n + 1) / 2, cnt = n;
    auto in = [&](uint64_t w, int32_t i) { return (kb >= 64 || w >> kb == kv) && i >> pb == pv; };
    while (cnt > kSplitRank) {
        if (tid < 256) hist[tid] = 0;
        __syncthreads();
        const bool pos = kb == 0;
        const int from = pos ? pb : kb, sh = from > 8 ? from - 8 : 0;
        const uint32_t mask = (1u << (from - sh)) - 1;
        for (int32_t i = tid; i < n; i += NT) {
            const uint64_t w = (uint64_t)keys[i] - (uint64_t)lo;
            if (in(w, i)) atomicAdd(&hist[(pos ? (uint32_t)(i >> sh) : (uint32_t)(w >> sh)) & mask], 1);
        }
        __syncthreads();
        int32_t h = 0, x = 0;
        if (tid < 256) {
            h = x = hist[tid];
            for (int d = 1; d < 32; d <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
                if (lane >= d) x += y;
            }
            if (lane == 31) wsum[warp] = x;
        }
        __syncthreads();
        if (tid < 256) {
            for (int w = 0; w < warp; ++w) x += wsum[w];
            if (x >= need && x - h < need) {
                s_bin = tid;
                s_need = need - (x - h);
                s_cnt = h;
            }
        }
        __syncthreads();
        need = s_need;
        cnt = s_cnt;
        if (pos) {
            pv = pv << (from - sh) | s_bin;
            pb = sh;
        } else {
            kv = kv << (from - sh) | (uint64_t)s_bin;
            kb = sh;
        }
    }
    if (tid == 0) s_fill = 0;
    __syncthreads();
    for (int32_t i = tid; i < n; i += NT) {
        const uint64_t w = (uint64_t)keys[i] - (uint64_t)lo;
        if (in(w, i)) {
            const int32_t j = atomicAdd(&s_fill, 1);
            cw[j] = w;
            cp[j] = i;
        }
    }
    __syncthreads();
    if (tid < cnt) {
        const uint64_t w = cw[tid];
        const int32_t p = cp[tid];
        int32_t below = 0;
        for (int j = 0; j < cnt; ++j) below += cw[j] < w || (cw[j] == w && cp[j] < p);
        if (below == need - 1) {
            s_w = w;
            s_p = p;
        }
    }
    __syncthreads();
    const uint64_t mw = s_w;
    const int32_t mp = s_p;
    for (int32_t i = tid; i < n; i += NT) {
        const uint64_t w = (uint64_t)keys[i] - (uint64_t)lo;
        child[members[i]] = 2 * c + (w < mw || (w == mw && i <= mp) ? 0 : 1);
    }
}

__global__ void k_gather(const int32_t* __restrict__ src, const int32_t* __restrict__ idx, int64_t n,
                         int32_t* __restrict__ dst)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) dst[i] = src[idx[i]];
}

__global__ void k_split_assign(const int32_t* __restrict__ order, const int32_t* __restrict__ cl,
                               const int32_t* __restrict__ start, int64_t T, int32_t* __restrict__ child,
                               int32_t* err)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= T) return;
    const int32_t c = cl[i];
    const int32_t size = start[c + 1] - start[c];
    if (size < 2) atomicOr(err, kErrEmpty);
    const int32_t rank = (int32_t)i - start[c];
    child[order[i]] = 2 * c + (rank < (size + 1) / 2 ? 0 : 1);
}

__global__ void k_children(int32_t K2, const double* __restrict__ frames, int32_t* __restrict__ parent,
                           double* __restrict__ fallback)
{
    int32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= K2) return;
    parent[c] = c >> 1;
    for (int i = 0; i < 9; ++i) fallback[9 * (int64_t)c + i] = frames[9 * (int64_t)(c >> 1) + i];
}

struct LevelObv {
    const uint64_t* obv[kMaxLevels];
    int32_t K[kMaxLevels];
};

// block per level: its total outer volume (whole numbers; a tree's total stays below 2^53)
__global__ void __launch_bounds__(256) k_level_totals(const LevelObv lv, uint64_t* __restrict__ out)
{
    const uint64_t* o = lv.obv[blockIdx.x];
    unsigned long long s = 0;
    for (int32_t i = threadIdx.x; i < lv.K[blockIdx.x]; i += 256) s += o[i];
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    __shared__ unsigned long long sh[8];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < 8; ++i) t += sh[i];
        out[blockIdx.x] = t;
    }
}

}  // namespace

// All levels in one launch and one copy: a copy and a synchronisation per
// level took 0.2 ms a score of nine levels, and a sweep scores its tree before
// and after every level.
obb_status tree_totals(obb_ctx* ctx, const obb_tree* tree, uint64_t* host)
{
    const int n = (int)tree->layers.size();
    if (n > kMaxLevels) return fail(ctx, OBB_ERR_STATE, "too many levels");
    LevelObv lv{};
    for (int i = 0; i < n; ++i) {
        lv.obv[i] = tree->layers[i]->d_obv;
        lv.K[i] = tree->layers[i]->K;
    }
    OBB_CK(ctx, ctx->tmp_d.reserve(sizeof(uint64_t) * kMaxLevels, ctx->stream));
    k_level_totals<<<n, 256, 0, ctx->stream>>>(lv, ctx->tmp_d.as<uint64_t>());
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    OBB_CK(ctx, cudaMemcpyAsync(host, ctx->tmp_d.p, sizeof(uint64_t) * n, cudaMemcpyDeviceToHost, ctx->stream));
    return check_device_error(ctx);
}

// Median split of every cluster of `up` into children 2c and 2c + 1; writes
// d_child[T].  Uses ctx->tmp_a for keys and sort buffers.  even: the clusters
// came from median splits, so none holds most of the triangles.
obb_status split_layer(obb_ctx* ctx, const obb_layer* up, int32_t* d_child, bool even)
{
    cudaStream_t s = ctx->stream;
    const obb_lattice* lat = up->lat;
    const int64_t T = up->T;
    const int32_t K = up->K;
    OBB_TRY(layer_members(ctx, const_cast<obb_layer*>(up)));   // brings the lists behind the handle up to date
    // Selection walks a cluster with one block: 36 us for one cluster of 10,000 triangles, 97 for 65,536 and 628 for
    // 524,288; the sorts take 151, 171 and 207 us (10,000, 65,536 and 524,288 triangles, any number of clusters).  So
    // up to 131,072 triangles however they are spread (173 against 178 us at worst), beyond that only where the
    // clusters are known to be of like size (524,288 triangles in 16 clusters: 61 against 209 us).
    if (T <= 131072 || (even && T <= 65536 * (int64_t)K)) {
        OBB_CK(ctx, ctx->tmp_a.reserve(sizeof(int64_t) * T, s));
        int64_t* keys = ctx->tmp_a.as<int64_t>();
        if (T > 2048 * (int64_t)(even ? K : 1))   // the cluster that may be met has that many
            k_split<1024><<<K, 1024, 0, s>>>(lat->d_fixed, lat->mesh->d_tris, up->d_members, up->d_start, up->d_q, keys,
                                             d_child, ctx->d_err);
        else
            k_split<256><<<K, 256, 0, s>>>(lat->d_fixed, lat->mesh->d_tris, up->d_members, up->d_start, up->d_q, keys,
                                           d_child, ctx->d_err);
        note_launch(ctx);
        OBB_CK(ctx, cudaGetLastError());
        return OBB_OK;   // an error found here is seen by the check of the layer made from d_child
    }
    OBB_CK(ctx, ctx->tmp_a.reserve(sizeof(int32_t) * T * 3 + sizeof(int64_t) * T * 2, s));
    int32_t* iota = ctx->tmp_a.as<int32_t>();
    int32_t* order1 = iota + T;
    int32_t* order2 = order1 + T;
    int64_t* keys = reinterpret_cast<int64_t*>(order2 + T);
    int64_t* keys_sorted = keys + T;
    int32_t* cl = reinterpret_cast<int32_t*>(keys_sorted);    // reused after the first sort
    int32_t* cl_sorted = cl + T;
    int end_bit = 1;
    while ((1 << end_bit) < K) ++end_bit;
    const unsigned gb = (unsigned)((T + 255) / 256);
    k_split_keys<<<gb, 256, 0, s>>>(lat->d_fixed, lat->mesh->d_tris, T, up->d_assign, up->d_q, keys, iota);
    note_launch(ctx);
    size_t b1 = 0, b2 = 0;
    OBB_CK(ctx, cub::DeviceRadixSort::SortPairs(nullptr, b1, keys, keys_sorted, iota, order1, (int)T, 0, 64, s));
    OBB_CK(ctx, cub::DeviceRadixSort::SortPairs(nullptr, b2, cl, cl_sorted, order1, order2, (int)T, 0, end_bit, s));
    OBB_CK(ctx, ctx->cub_tmp.reserve(b1 > b2 ? b1 : b2, s));
    auto sort1 = [&](cudaStream_t cs) {
        size_t bb = ctx->cub_tmp.bytes;
        return cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, bb, keys, keys_sorted, iota, order1, (int)T, 0, 64, cs);
    };
    OBB_CK(ctx, sort1(s));
    note_launch(ctx, captured_launches(ctx, T, 1000 + 64, sort1));
    k_gather<<<gb, 256, 0, s>>>(up->d_assign, order1, T, cl);
    note_launch(ctx);
    auto sort2 = [&](cudaStream_t cs) {
        size_t bb = ctx->cub_tmp.bytes;
        return cub::DeviceRadixSort::SortPairs(ctx->cub_tmp.p, bb, cl, cl_sorted, order1, order2, (int)T, 0, end_bit,
                                               cs);
    };
    OBB_CK(ctx, sort2(s));
    note_launch(ctx, captured_launches(ctx, T, end_bit, sort2));
    k_split_assign<<<gb, 256, 0, s>>>(order2, cl_sorted, up->d_start, T, d_child, ctx->d_err);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return check_device_error(ctx);
}

obb_status build_tree(obb_ctx* ctx, const obb_lattice* lat, const obb_tree_opts* opts, obb_tree* tree)
{
    cudaStream_t s = ctx->stream;
    const int64_t T = lat->mesh->nt;
    const int depth = opts->depth;
    if (depth < 0 || depth > 20) return fail(ctx, OBB_ERR_ARG, "depth must be in [0, 20]");
    if ((int64_t(1) << depth) > T) return fail(ctx, OBB_ERR_EMPTY_CLUSTER, "fewer triangles than leaves");
    tree->ctx = ctx;
    tree->lat = lat;
    const int64_t Kmax = int64_t(1) << depth;
    OBB_CK(ctx, ctx->tmp_c.reserve(sizeof(int32_t) * T, s));
    OBB_CK(ctx, ctx->tmp_b.reserve(sizeof(int32_t) * Kmax + 64 + 9 * sizeof(double) * Kmax, s));
    int32_t* child = ctx->tmp_c.as<int32_t>();
    int32_t* parent = ctx->tmp_b.as<int32_t>();
    double* fallback = reinterpret_cast<double*>(ctx->tmp_b.as<char>() + ((sizeof(int32_t) * Kmax + 63) / 64) * 64);

    // root: every triangle in cluster 0, frame from the covariance
    OBB_CK(ctx, cudaMemsetAsync(child, 0, sizeof(int32_t) * T, s));
    OBB_CK(ctx, cudaMemsetAsync(parent, 0, sizeof(int32_t), s));
    obb_layer* root = nullptr;
    OBB_TRY(layer_create(ctx, lat, child, parent, 1, nullptr, nullptr, &root));
    tree->layers.push_back(root);
    obb_step_opts so{opts->rounds, opts->refit, 0, 0};
    for (int lev = 1; lev <= depth; ++lev) {
        obb_layer* up = tree->layers.back();
        OBB_TRY(split_layer(ctx, up, child, true));
        const int32_t K2 = 2 * up->K;
        k_children<<<(K2 + 127) / 128, 128, 0, s>>>(K2, up->d_frames, parent, fallback);
        note_launch(ctx);
        OBB_CK(ctx, cudaGetLastError());
        obb_layer* L = nullptr;
        OBB_TRY(layer_create(ctx, lat, child, parent, K2, nullptr, fallback, &L));
        tree->layers.push_back(L);
        for (int it = 0; it < opts->iters; ++it) {
            obb_step_stats st{};
            OBB_TRY(lloyd_step(ctx, L, &so, &st));
            if (st.moves == 0 && st.refits_accepted == 0) break;
        }
    }
    return OBB_OK;
}

}  // namespace obbv
