// Mesh upload and validation on the device (the closed mesh X of Sec. 3,
// Definition 1): every coordinate finite, every index in range, no triangle
// with a repeated vertex, and every undirected edge shared by exactly two
// triangles.  The pairing of the edges' two sides is also the triangle
// adjacency (triangle across edge (v_e, v_e+1)).
//
// The 3T half-edges are bucketed by their endpoint of smaller degree (the fan
// around a vertex of any degree then spreads over its rim), one bucket a
// vertex in no particular order, and every half-edge looks for its partner
// among the few in its bucket:
//   k_mesh_degrees  degrees (and the vertices' finiteness);
//   k_mesh_ranks    bucket sizes, every half-edge's place in its bucket;
//   k_mesh_starts   bucket starts: a block's scan and one atomic;
//   k_mesh_buckets  (other endpoint, half-edge) at its place;
//   k_mesh_pair     the partner: exactly one other half-edge of the bucket
//                   with the same other endpoint.
// Sorting the edge keys instead moves every key and slot five times: 2M
// triangles 343 us of kernels, the buckets 133 us (17 + 29 + 6 + 27 + 54; the
// gathers of the last three bound them).
#include <string>

#include "internal.h"

namespace obbv {
namespace {

enum { kMeshNonFinite = 1, kMeshRange = 2, kMeshRepeated = 4, kMeshEdge = 8 };

__global__ void k_mesh_degrees(const float* __restrict__ V, int64_t n3, const int32_t* __restrict__ F, int64_t nt,
                               int64_t nv, int32_t* __restrict__ deg, int32_t* __restrict__ flags)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
    bool finite = true;
    for (int64_t i = t; i < n3; i += threads) finite &= isfinite(V[i]);
    int32_t f = finite ? 0 : kMeshNonFinite;
    int32_t v[3] = {-1, -1, -1};
    if (t < nt) {
        for (int e = 0; e < 3; ++e) {
            v[e] = F[3 * t + e];
            if (v[e] < 0 || v[e] >= nv) f |= kMeshRange;
        }
        if (v[0] == v[1] || v[1] == v[2] || v[2] == v[0]) f |= kMeshRepeated;
    }
    const int lane = threadIdx.x & 31;
    for (int e = 0; e < 3; ++e) {
        const bool on = t < nt && v[e] >= 0 && v[e] < nv;
        // Triangles of a fan lie side by side and add to one word, one after another: a corner that the whole warp
        // shares adds once (two hubs of 200,000 triangles each: a call 376 -> 134 us; other meshes of 2M 17 -> 19 here)
        int same = 0;
        __match_all_sync(0xffffffffu, v[e], &same);
        if (same) {
            const int n = __popc(__ballot_sync(0xffffffffu, on));
            if (lane == 0 && n) atomicAdd(&deg[v[e]], n);
        } else if (on) {
            atomicAdd(&deg[v[e]], 1);
        }
    }
    if (f) atomicOr(flags, f);
}

// endpoints of half-edge i; false: an index out of range (reported above)
__device__ __forceinline__ bool half_edge(const int32_t* __restrict__ F, int64_t i, int64_t nv, int32_t& a, int32_t& b)
{
    const int64_t t = i / 3;
    const int e = (int)(i - 3 * t);
    a = __ldg(F + i);
    b = __ldg(F + 3 * t + (e == 2 ? 0 : e + 1));
    return a >= 0 && a < nv && b >= 0 && b < nv;
}

// rank[i]: twice the place of half-edge i in its bucket, plus 1 if the
// bucket is its second endpoint's; both halves of an edge choose the same
// endpoint: the one of smaller degree, then of smaller index
__global__ void k_mesh_ranks(const int32_t* __restrict__ F, int64_t ne, int64_t nv, const int32_t* __restrict__ deg,
                             int32_t* __restrict__ size, uint32_t* __restrict__ rank)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int32_t a, b;
    if (i >= ne || !half_edge(F, i, nv, a, b)) return;
    const int32_t da = __ldg(deg + a), db = __ldg(deg + b);
    const bool second = db < da || (db == da && b < a);
    rank[i] = 2u * (uint32_t)atomicAdd(&size[second ? b : a], 1) + (second ? 1u : 0u);
}

__global__ void __launch_bounds__(256) k_mesh_starts(const int32_t* __restrict__ size, int64_t nv,
                                                     uint32_t* __restrict__ start, uint32_t* __restrict__ total)
{
    __shared__ uint32_t ws[8], base;
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t n = v < nv ? (uint32_t)((size[v] + 1) & ~1) : 0u;   // items are read in pairs
    uint32_t x = n;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int i = 0; i < 8; ++i) {
            const uint32_t c = ws[i];
            ws[i] = t;
            t += c;
        }
        base = t ? atomicAdd(total, t) : 0u;
    }
    __syncthreads();
    if (v < nv) start[v] = base + ws[w] + x - n;
}

__global__ void k_mesh_buckets(const int32_t* __restrict__ F, int64_t ne, int64_t nv,
                               const uint32_t* __restrict__ rank, const uint32_t* __restrict__ start,
                               uint2* __restrict__ item)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int32_t a, b;
    if (i >= ne || !half_edge(F, i, nv, a, b)) return;
    const uint32_t r = rank[i];
    const bool second = r & 1u;
    item[__ldg(start + (second ? b : a)) + (r >> 1)] = make_uint2((uint32_t)(second ? a : b), (uint32_t)i);
}

__device__ __forceinline__ unsigned long long edge_key(int32_t a, int32_t b, int B)
{
    return ((unsigned long long)min(a, b) << B) | (unsigned long long)max(a, b);
}

__global__ void k_mesh_pair(const int32_t* __restrict__ F, int64_t ne, int64_t nv, int B,
                            const uint32_t* __restrict__ rank, const uint32_t* __restrict__ start,
                            const int32_t* __restrict__ size, const uint2* __restrict__ item,
                            int32_t* __restrict__ adj, unsigned long long* __restrict__ bad,
                            int32_t* __restrict__ flags)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int32_t a, b;
    if (i >= ne || !half_edge(F, i, nv, a, b)) return;
    const bool second = rank[i] & 1u;
    const int32_t v = second ? b : a;
    const uint32_t other = (uint32_t)(second ? a : b), b0 = __ldg(start + v), b1 = b0 + (uint32_t)__ldg(size + v);
    int found = 0;
    uint32_t partner = 0;
    for (uint32_t j = b0; j < b1 && found < 2; j += 4) {   // two others are too many already
        uint4 x[2];   // two items each; past the bucket: this half-edge itself
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            x[u] = make_uint4(0u, (uint32_t)i, 0u, (uint32_t)i);
            if (j + 2 * u < b1) x[u] = __ldg(reinterpret_cast<const uint4*>(item + j + 2 * u));
            if (j + 2 * u + 1 >= b1) x[u].w = (uint32_t)i;
            if (x[u].x == other && x[u].y != (uint32_t)i) {
                partner = x[u].y;
                ++found;
            }
            if (x[u].z == other && x[u].w != (uint32_t)i) {
                partner = x[u].w;
                ++found;
            }
        }
    }
    if (found == 1) {
        adj[i] = (int32_t)(partner / 3u);
    } else {
        atomicOr(flags, kMeshEdge);
        atomicMin(bad, edge_key(a, b, B));
    }
}

__global__ void k_mesh_count_key(const int32_t* __restrict__ F, int64_t ne, int64_t nv, int B,
                                 const unsigned long long* __restrict__ bad, int32_t* __restrict__ count)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    int32_t a, b;
    if (i < ne && half_edge(F, i, nv, a, b) && edge_key(a, b, B) == *bad) atomicAdd(count, 1);
}

}  // namespace

obb_status mesh_upload(obb_ctx* ctx, const float* verts, int64_t nv, const int32_t* tris, int64_t nt, obb_mesh* m)
{
    cudaStream_t s = ctx->stream;
    const int64_t ne = 3 * nt;
    OBB_CK(ctx, pool_alloc((void**)&m->d_verts, sizeof(float) * 3 * nv, s));
    OBB_CK(ctx, pool_alloc((void**)&m->d_tris, sizeof(int32_t) * ne, s));
    OBB_CK(ctx, pool_alloc((void**)&m->d_adj, sizeof(int32_t) * ne, s));
    OBB_CK(ctx, cudaMemcpyAsync(m->d_verts, verts, sizeof(float) * 3 * nv, cudaMemcpyHostToDevice, s));
    OBB_CK(ctx, cudaMemcpyAsync(m->d_tris, tris, sizeof(int32_t) * ne, cudaMemcpyHostToDevice, s));
    int B = 1;   // bits of a vertex index
    while (B < 31 && (int64_t(1) << B) < nv) ++B;
    // scratch: the zeroed words (degrees, bucket sizes, flags, their total, the bad key's count), the smallest bad
    // key, bucket starts, half-edges' places, bucket items
    auto up = [](size_t n) { return (n + 255) / 256 * 256; };
    const size_t vb = up(sizeof(int32_t) * nv), eb = up(sizeof(int32_t) * ne);
    OBB_CK(ctx, ctx->tmp_a.reserve(3 * vb + 512 + eb + sizeof(uint2) * (ne + nv), s));
    char* base = ctx->tmp_a.as<char>();
    int32_t* deg = reinterpret_cast<int32_t*>(base);
    int32_t* size = reinterpret_cast<int32_t*>(base + vb);
    int32_t* flags = reinterpret_cast<int32_t*>(base + 2 * vb);
    uint32_t* total = reinterpret_cast<uint32_t*>(base + 2 * vb + 64);
    int32_t* bad_count = reinterpret_cast<int32_t*>(base + 2 * vb + 128);
    unsigned long long* bad = reinterpret_cast<unsigned long long*>(base + 2 * vb + 256);
    uint32_t* start = reinterpret_cast<uint32_t*>(base + 2 * vb + 512);
    uint32_t* rank = reinterpret_cast<uint32_t*>(base + 3 * vb + 512);
    uint2* item = reinterpret_cast<uint2*>(base + 3 * vb + 512 + eb);
    OBB_CK(ctx, cudaMemsetAsync(base, 0, 2 * vb + 256, s));
    OBB_CK(ctx, cudaMemsetAsync(bad, 0xff, sizeof(unsigned long long), s));
    const unsigned ge = (unsigned)((ne + 255) / 256);
    k_mesh_degrees<<<(unsigned)((nt + 255) / 256), 256, 0, s>>>(m->d_verts, 3 * nv, m->d_tris, nt, nv, deg, flags);
    k_mesh_ranks<<<ge, 256, 0, s>>>(m->d_tris, ne, nv, deg, size, rank);
    k_mesh_starts<<<(unsigned)((nv + 255) / 256), 256, 0, s>>>(size, nv, start, total);
    k_mesh_buckets<<<ge, 256, 0, s>>>(m->d_tris, ne, nv, rank, start, item);
    k_mesh_pair<<<ge, 256, 0, s>>>(m->d_tris, ne, nv, B, rank, start, size, item, m->d_adj, bad, flags);
    note_launch(ctx, 5);
    OBB_CK(ctx, cudaGetLastError());
    int32_t* h = reinterpret_cast<int32_t*>(host_stats(ctx));
    OBB_CK(ctx, cudaMemcpyAsync(h, flags, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    OBB_CK(ctx, cudaStreamSynchronize(s));
    const int32_t f = h[0];
    if (f & kMeshNonFinite) return fail(ctx, OBB_ERR_ARG, "non-finite vertex coordinate");
    if (f & kMeshRange) return fail(ctx, OBB_ERR_ARG, "triangle index out of range");
    if (f & kMeshRepeated) return fail(ctx, OBB_ERR_NOT_WATERTIGHT, "triangle with a repeated vertex");
    if (f & kMeshEdge) {
        k_mesh_count_key<<<ge, 256, 0, s>>>(m->d_tris, ne, nv, B, bad, bad_count);
        note_launch(ctx);
        unsigned long long hb = 0;
        OBB_CK(ctx, cudaMemcpyAsync(&hb, bad, sizeof(hb), cudaMemcpyDeviceToHost, s));
        OBB_CK(ctx, cudaMemcpyAsync(h + 1, bad_count, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
        OBB_CK(ctx, cudaStreamSynchronize(s));
        return fail(ctx, OBB_ERR_NOT_WATERTIGHT,
                    "edge (" + std::to_string(hb >> B) + ", " + std::to_string(hb & ((1ull << B) - 1)) + ") is shared by " +
                        std::to_string(h[1]) + " triangles (need exactly 2)");
    }
    return OBB_OK;
}

}  // namespace obbv
