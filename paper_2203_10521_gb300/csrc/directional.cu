// The paper's own outer-volume estimator (Sec. 4.1, Eq. 9-10), restated as
// CUDA ray casting instead of cube-map rasterisation.
//
// From the box centre o, one ray per texel of a 6 x m x m cube map (direction
// through the texel centre, weight = the texel's exact solid angle).  Along a
// ray the mesh crossings at distances r_i < r_e (r_e = where the ray leaves the
// box) carry sign s_i = +1 when the ray leaves the solid (n . w > 0) and -1
// when it enters (the convention of Fig. 1a).  With chi(o) = 1 when o is
// inside the solid, the inside length of the segment is
//   l_in = sum_i s_i r_i + chi(p_e) r_e,   chi(p_e) = chi(o) - sum_i s_i,
// and the cone volumes give
//   V_out(w) = dOmega / 3 (r_e^3 - sum_i s_i r_i^3 - chi(p_e) r_e^3).
// The estimate is the sum over texels.  chi(o) is the signed crossing count of
// a ray from o to infinity (outward-oriented closed mesh).  FP32 arithmetic,
// Moeller-Trumbore intersections against every triangle that the ray's texel
// can meet.
#include <cooperative_groups.h>

#include <algorithm>

#include "internal.h"

namespace obbv {
namespace {

__device__ __forceinline__ bool ray_tri(const float3 o, const float3 d, const float3 a, const float3 b,
                                        const float3 c, float& t, float& sgn)
{
    const float3 e1 = make_float3(b.x - a.x, b.y - a.y, b.z - a.z);
    const float3 e2 = make_float3(c.x - a.x, c.y - a.y, c.z - a.z);
    const float3 p = make_float3(d.y * e2.z - d.z * e2.y, d.z * e2.x - d.x * e2.z, d.x * e2.y - d.y * e2.x);
    const float det = e1.x * p.x + e1.y * p.y + e1.z * p.z;
    if (fabsf(det) < 1e-20f) return false;
    const float inv = 1.f / det;
    const float3 s = make_float3(o.x - a.x, o.y - a.y, o.z - a.z);
    const float u = (s.x * p.x + s.y * p.y + s.z * p.z) * inv;
    if (u < 0.f || u > 1.f) return false;
    const float3 q = make_float3(s.y * e1.z - s.z * e1.y, s.z * e1.x - s.x * e1.z, s.x * e1.y - s.y * e1.x);
    const float v = (d.x * q.x + d.y * q.y + d.z * q.z) * inv;
    if (v < 0.f || u + v > 1.f) return false;
    t = (e2.x * q.x + e2.y * q.y + e2.z * q.z) * inv;
    if (t <= 0.f) return false;
    // outward normal e1 x e2: leaving the solid when it points along d (det = -(e1 x e2) . d)
    sgn = det < 0.f ? 1.f : -1.f;
    return true;
}

__device__ __forceinline__ float texel_solid_angle(float u0, float u1, float v0, float v1)
{
    auto F = [](float u, float v) { return atan2f(u * v, sqrtf(u * u + v * v + 1.f)); };
    return F(u1, v1) - F(u0, v1) - F(u1, v0) + F(u0, v0);
}

// direction through the point (uc, vc) of a face, normalised
__device__ __forceinline__ float3 texel_dir(int face, float uc, float vc)
{
    const int axis = face >> 1;
    const float sgn = (face & 1) ? -1.f : 1.f;
    const float x = axis == 0 ? sgn : axis == 1 ? vc : uc;
    const float y = axis == 0 ? uc : axis == 1 ? sgn : vc;
    const float z = axis == 0 ? vc : axis == 1 ? uc : sgn;
    const float nrm = rsqrtf(__fmaf_rn(z, z, __fmaf_rn(x, x, __fmul_rn(y, y))));
    return make_float3(x * nrm, y * nrm, z * nrm);
}

constexpr int kDirThreads = 512;
constexpr int kDirTexels = 2048;    // texels a block holds at once (96 KB: two blocks on an SM)
constexpr int kDirHits = 3;         // crossings a texel keeps one by one
constexpr int kDirQueue = 1024;     // triangles with many texels, shared out over whole warps
constexpr int kDirInline = 64;      // texels a triangle may have without being queued

// A texel's ray while the triangles are projected onto it: its exit
// distance, the number and the signed number of crossings before it, and the
// first kDirHits to arrive (triangle, signed distance), whose cubes are added
// in FP32 in the order of the triangles at the end.  With more crossings the
// cubes are added in fixed point, 37 bits below the exit distance's cube:
// whole numbers, so neither sum depends on the order of arrival.  A cube is
// then off by its own FP32 rounding and 2^-38 of the power of two below the
// exit cube, so n of them add less than n 2^-38 of the exit cube; an FP32 sum
// adds up to 2^-24 of every partial sum.  (An exit cube that is no normal
// number, of a box below 10^-12 or beyond 10^12 in size, takes none.)
struct DirTexel {
    unsigned long long s3;
    float re;
    int32_t n, s1;
    int32_t t[kDirHits];
    float q[kDirHits];
};

struct DirItem {
    int32_t t;
    uint16_t face;
    uint8_t u0, u1, v0, v1;
};

// exponent of the exit distance's cube; kNoCube when it is no normal number (the ray then takes no cubes)
constexpr int kNoCube = 1000;
__device__ __forceinline__ int cube_exponent(float re)
{
    const float re3 = re * re * re;
    const int e = (int)(__float_as_uint(re3) >> 23) - 127;   // sign and exponent: > 127 when negative
    return e > -127 && e < 127 ? e : kNoCube;
}

// (q |q|^2) in fixed point for a ray of cube exponent e: times 2^-e, then 2^37, both exact
__device__ __forceinline__ unsigned long long fixed_cube(float q, int e)
{
    if (e == kNoCube) return 0ull;
    return (unsigned long long)__float2ll_rn(q * q * q * __uint_as_float((uint32_t)(127 - e) << 23) * 0x1p37f);
}

struct DirTri {
    float3 a, b, c;
};

__device__ __forceinline__ DirTri dir_load(const float* __restrict__ V, const int32_t* __restrict__ F, int64_t t)
{
    const float* a = V + 3 * (int64_t)__ldg(F + 3 * t);
    const float* b = V + 3 * (int64_t)__ldg(F + 3 * t + 1);
    const float* c = V + 3 * (int64_t)__ldg(F + 3 * t + 2);
    return DirTri{make_float3(__ldg(a), __ldg(a + 1), __ldg(a + 2)), make_float3(__ldg(b), __ldg(b + 1), __ldg(b + 2)),
                  make_float3(__ldg(c), __ldg(c + 1), __ldg(c + 2))};
}

// one texel's ray against triangle t
__device__ __forceinline__ void dir_test(const float3 o, int32_t t, const DirTri& T, int face, float uc, float vc,
                                         DirTexel* __restrict__ x)
{
    float tt, sg;
    if (ray_tri(o, texel_dir(face, uc, vc), T.a, T.b, T.c, tt, sg) && tt < x->re) {
        atomicAdd(&x->s1, sg > 0.f ? 1 : -1);
        const int i = atomicAdd(&x->n, 1);
        if (i < kDirHits) {
            x->t[i] = t;
            x->q[i] = sg * tt;
        } else {
            atomicAdd(&x->s3, fixed_cube(sg * tt, cube_exponent(x->re)));
        }
    }
}

// the signed sum of a ray's cubed crossings
__device__ __forceinline__ double sum_cubes(DirTexel y)
{
    if (y.n > kDirHits) {
        const int e = cube_exponent(y.re);
        unsigned long long s = y.s3;
#pragma unroll
        for (int i = 0; i < kDirHits; ++i) s += fixed_cube(y.q[i], e);
        return e != kNoCube ? (double)(long long)s * __hiloint2double((e - 37 + 1023) << 20, 0) : 0.0;
    }
    // in triangle order, which a comparison network of three gives
    static_assert(kDirHits == 3, "three crossings are sorted");
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (i >= y.n) {
            y.t[i] = INT32_MAX;
            y.q[i] = 0.f;
        }
    auto order = [&](int a, int b) {
        if (y.t[a] > y.t[b]) {
            const int32_t t = y.t[a];
            const float q = y.q[a];
            y.t[a] = y.t[b];
            y.q[a] = y.q[b];
            y.t[b] = t;
            y.q[b] = q;
        }
    };
    order(0, 1);
    order(1, 2);
    order(0, 1);
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 3; ++i) s = __fmaf_rn(__fmul_rn(y.q[i], fabsf(y.q[i])), fabsf(y.q[i]), s);
    return (double)s;
}

// The texels [r0, r1) x [0, m) of a face that a triangle can meet, from its
// vertices relative to the box centre; false if none.  Every texel whose ray
// meets the triangle is among them: the ranges are those of the projected
// vertices, widened by 0.02 texels + 1e-5 (the projection's rounding is
// below 1e-6), and a triangle that reaches behind the centre's plane and is
// not outside one of the face's four side planes takes the whole face.
__device__ __forceinline__ bool dir_rect(const float3 A, const float3 B, const float3 C, int face, int m, int r0,
                                         int r1, int& u0, int& u1, int& v0, int& v1)
{
    const int axis = face >> 1;
    const float sgn = (face & 1) ? -1.f : 1.f;
    auto pick = [&](const float3& p, float& w, float& x, float& y) {
        w = sgn * (axis == 0 ? p.x : axis == 1 ? p.y : p.z);
        x = axis == 0 ? p.y : axis == 1 ? p.z : p.x;
        y = axis == 0 ? p.z : axis == 1 ? p.x : p.y;
    };
    float wa, xa, ya, wb, xb, yb, wc, xc, yc;
    pick(A, wa, xa, ya);
    pick(B, wb, xb, yb);
    pick(C, wc, xc, yc);
    if (fmaxf(wa, fmaxf(wb, wc)) <= 0.f) return false;
    u0 = 0;
    u1 = m - 1;
    v0 = r0;
    v1 = r1 - 1;
    if (fminf(wa, fminf(wb, wc)) > 0.f) {
        const float ia = __fdividef(1.f, wa), ib = __fdividef(1.f, wb), ic = __fdividef(1.f, wc);
        const float h = 0.5f * m, pad = 0.02f + 1e-5f * h;
        const float ua = xa * ia, ub = xb * ib, uc = xc * ic, va = ya * ia, vb = yb * ib, vc = yc * ic;
        const float fu0 = (fminf(ua, fminf(ub, uc)) + 1.f) * h - pad, fu1 = (fmaxf(ua, fmaxf(ub, uc)) + 1.f) * h + pad;
        const float fv0 = (fminf(va, fminf(vb, vc)) + 1.f) * h - pad, fv1 = (fmaxf(va, fmaxf(vb, vc)) + 1.f) * h + pad;
        // texel i's ray passes at i + 1/2
        if (fu1 < 0.5f || fu0 > m - 0.5f || fv1 < r0 + 0.5f || fv0 > r1 - 0.5f) return false;
        u0 = max(u0, (int)ceilf(fmaxf(fu0, 0.f) - 0.5f));
        u1 = min(u1, (int)floorf(fminf(fu1, (float)m) - 0.5f));
        v0 = max(v0, (int)ceilf(fmaxf(fv0, 0.f) - 0.5f));
        v1 = min(v1, (int)floorf(fminf(fv1, (float)m) - 0.5f));
        return u0 <= u1 && v0 <= v1;
    }
    // outside a side plane |x| <= w or |y| <= w, with a margin far above the rounding
    auto out = [](float xa, float wa, float xb, float wb, float xc, float wc) {
        return xa - wa > 1e-4f * (fabsf(xa) + fabsf(wa)) && xb - wb > 1e-4f * (fabsf(xb) + fabsf(wb)) &&
               xc - wc > 1e-4f * (fabsf(xc) + fabsf(wc));
    };
    return !(out(xa, wa, xb, wb, xc, wc) || out(-xa, wa, -xb, wb, -xc, wc) || out(ya, wa, yb, wb, yc, wc) ||
             out(-ya, wa, -yb, wb, -yc, wc));
}

// A cluster of G = 1, 2, 3 or 6 blocks per box, 6 / G faces a block.  Testing
// every ray against every triangle is 6 m^2 nt tests a box, bound by FP32
// issue (64 boxes, 10k triangles, m = 32: 42.2 ms); a triangle meets only the
// rays inside its projection, so a thread projects a triangle onto the faces
// and only the texels it covers are tested, with the same ray-triangle test,
// each ray keeping its sums in shared memory (the same call: 0.066 ms).  What
// is left is the walk over the mesh (gathers from L2) and the boxes near the
// surface, where a few triangles cover many texels.
// - Triangles beyond the box's farthest exit are left out.
// - The tests of a warp's 32 triangles are dealt out one a lane (a lane
//   walking its own triangle's texels leaves most of the warp idle: 0.125 ms),
//   and triangles over more than kDirInline texels are queued and shared out
//   over all the block's warps (32 or 64: equal; 128: slower).
// - A block takes its faces' texels in chunks of at most kDirTexels (48 bytes
//   each) and walks the mesh once per chunk, so every m fits.
// - The blocks of a cluster share the crossings of the chi ray and their
//   partial sums through distributed shared memory: no scratch, one launch.
__global__ void __launch_bounds__(kDirThreads, 2) k_directional(const float* __restrict__ V,
                                                                const int32_t* __restrict__ Fi, int64_t nt,
                                                                const obb_box* __restrict__ boxes, int32_t m,
                                                                int32_t G, double* __restrict__ out)
{
    extern __shared__ __align__(16) unsigned char dir_smem[];
    DirTexel* tx = reinterpret_cast<DirTexel*>(dir_smem);
    __shared__ DirItem queue[kDirQueue];
    __shared__ float mid[256];             // texel centres along u and v (m <= 256)
    __shared__ int32_t queued, chi;
    __shared__ int32_t reach;              // bits of the chunk's largest exit distance (positive floats order as ints)
    __shared__ double part[kDirThreads / 32];
    __shared__ double block_sum;
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const obb_box B = boxes[blockIdx.x / G];
    const float3 o = make_float3(B.c[0], B.c[1], B.c[2]);
    const float3 ax[3] = {make_float3(B.axis0[0], B.axis0[1], B.axis0[2]),
                          make_float3(B.axis1[0], B.axis1[1], B.axis1[2]),
                          make_float3(B.axis0[1] * B.axis1[2] - B.axis0[2] * B.axis1[1],
                                      B.axis0[2] * B.axis1[0] - B.axis0[0] * B.axis1[2],
                                      B.axis0[0] * B.axis1[1] - B.axis0[1] * B.axis1[0])};
    const float size = fabsf(o.x) + fabsf(o.y) + fabsf(o.z);
    const bool finite = size < 3.0e38f;    // no ray from another centre meets anything
    const int F = 6 / G, f0 = rank * F;
    // a chunk: whole faces while they fit, else rows of one face
    const int rows = max(1, min(m, kDirTexels / m));
    const int bands = (m + rows - 1) / rows;
    const int faces = bands > 1 ? 1 : max(1, min(F, kDirTexels / (m * m)));
    double vol = 0.0;
    if (tid == 0) chi = 0;
    if (tid < m) {
        const float a = -1.f + 2.f * tid / m, b = -1.f + 2.f * (tid + 1) / m;
        mid[tid] = 0.5f * (a + b);
    }
    for (int c = 0; c < ((F + faces - 1) / faces) * bands; ++c) {
        const int fa = f0 + (c / bands) * faces, fb = min(fa + faces, f0 + F);
        const int r0 = (c % bands) * rows, r1 = min(m, r0 + rows), per = (r1 - r0) * m, texels = (fb - fa) * per;
        if (tid == 0) {
            queued = 0;
            reach = 0;
        }
        __syncthreads();
        float far = 0.f;
        for (int x = tid; x < texels; x += kDirThreads) {
            const int r = x % per;
            const float3 d = texel_dir(fa + x / per, mid[r % m], mid[r0 + r / m]);
            // exit distance from the box (centre o): min_a half_a / |axis_a . d|
            float re = 3.0e38f;
            for (int a = 0; a < 3; ++a) {
                const float q = fabsf(ax[a].x * d.x + ax[a].y * d.y + ax[a].z * d.z);
                if (q > 0.f) re = fminf(re, B.half[a] / q);
            }
            tx[x].s3 = 0;
            tx[x].re = re;
            tx[x].n = tx[x].s1 = 0;
            far = fmaxf(far, re);
        }
        atomicMax(&reach, __float_as_int(far));
        __syncthreads();
        // |coordinate| of a crossing before any ray's exit (rays have length 1 to 1e-6), relative to the centre
        const float R = __int_as_float(reach) * 1.0001f;
        int32_t n = 0;
        for (int64_t t0 = 32 * warp; t0 < nt && finite; t0 += kDirThreads) {   // warp-uniform
            const int64_t t = t0 + lane;
            const bool live = t < nt;
            const DirTri T = dir_load(V, Fi, live ? t : t0);
            if (c == 0 && live && (int)((t0 >> 5) % G) == rank) {
                // chi(o): signed crossings of a ray from o towards a fixed generic direction
                float tt, sg;
                if (ray_tri(o, make_float3(0.5773502f, 0.5773503f, 0.5773502f), T.a, T.b, T.c, tt, sg))
                    n += sg > 0.f ? 1 : -1;
            }
            const float3 A = make_float3(T.a.x - o.x, T.a.y - o.y, T.a.z - o.z);
            const float3 Bv = make_float3(T.b.x - o.x, T.b.y - o.y, T.b.z - o.z);
            const float3 C = make_float3(T.c.x - o.x, T.c.y - o.y, T.c.z - o.z);
            const bool near = live && !(fminf(A.x, fminf(Bv.x, C.x)) > R || fmaxf(A.x, fmaxf(Bv.x, C.x)) < -R ||
                                        fminf(A.y, fminf(Bv.y, C.y)) > R || fmaxf(A.y, fmaxf(Bv.y, C.y)) < -R ||
                                        fminf(A.z, fminf(Bv.z, C.z)) > R || fmaxf(A.z, fmaxf(Bv.z, C.z)) < -R);
            if (!__any_sync(0xffffffffu, near)) continue;
            for (int face = fa; face < fb; ++face) {
                int u0 = 0, u1 = 0, v0 = 0, v1 = 0, cnt = 0;
                if (near && dir_rect(A, Bv, C, face, m, r0, r1, u0, u1, v0, v1)) cnt = (u1 - u0 + 1) * (v1 - v0 + 1);
                if (cnt > kDirInline) {
                    const int q = atomicAdd(&queued, 1);
                    if (q < kDirQueue) {
                        queue[q] = DirItem{(int32_t)t, (uint16_t)face, (uint8_t)u0, (uint8_t)u1, (uint8_t)v0,
                                           (uint8_t)v1};
                        cnt = 0;
                    }
                }
                // the warp's (triangle, texel) pairs, dealt out one a lane
                int inc = cnt;
                for (int off = 1; off < 32; off <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, off);
                    if (lane >= off) inc += y;
                }
                const int total = __shfl_sync(0xffffffffu, inc, 31);
                const int first = inc - cnt;
                const uint32_t rect = (uint32_t)u0 | (uint32_t)v0 << 8 | (uint32_t)(u1 - u0) << 16;
                DirTexel* base = tx + (face - fa) * per - r0 * m;
                for (int i0 = 0; i0 < total; i0 += 32) {
                    const int i = i0 + lane;
                    int src = 0;   // the first lane whose pairs end beyond i
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(0xffffffffu, inc, src + step - 1) <= i) src += step;
                    const uint32_t rc = __shfl_sync(0xffffffffu, rect, src);
                    const int e = i - __shfl_sync(0xffffffffu, first, src);
                    if (i >= total) continue;
                    const int nu = (int)(rc >> 16) + 1, row = e / nu;
                    const int iu = (int)(rc & 0xff) + e - row * nu, iv = (int)(rc >> 8 & 0xff) + row;
                    dir_test(o, (int32_t)(t0 + src), dir_load(V, Fi, t0 + src), face, mid[iu], mid[iv], base + iv * m + iu);
                }
            }
        }
        if (c == 0) {
            n = __reduce_add_sync(0xffffffffu, n);
            if (lane == 0 && n) atomicAdd(&chi, n);
        }
        __syncthreads();
        const int items = min(queued, kDirQueue);
        for (int q = warp; q < items; q += kDirThreads / 32) {
            const DirItem it = queue[q];
            const DirTri T = dir_load(V, Fi, it.t);
            DirTexel* base = tx + (it.face - fa) * per - r0 * m;
            const int nu = it.u1 - it.u0 + 1, cnt = nu * (it.v1 - it.v0 + 1);
            for (int i = lane; i < cnt; i += 32) {
                const int iu = it.u0 + i % nu, iv = it.v0 + i / nu;
                dir_test(o, it.t, T, it.face, mid[iu], mid[iv], base + iv * m + iu);
            }
        }
        // chi of the whole cluster, complete after every block's first walk
        if (c == 0) cluster.sync();
        else __syncthreads();
        int32_t chi_all = 0;
        for (int g = 0; g < G; ++g) chi_all += *cluster.map_shared_rank(&chi, g);
        const float chi_o = (float)chi_all;
        for (int x = tid; x < texels; x += kDirThreads) {
            const DirTexel y = tx[x];
            const int r = x % per, iu = r % m, iv = r0 + r / m;
            const float u0 = -1.f + 2.f * iu / m, u1 = -1.f + 2.f * (iu + 1) / m;
            const float v0 = -1.f + 2.f * iv / m, v1 = -1.f + 2.f * (iv + 1) / m;
            const float chi_e = chi_o - (float)y.s1, re3 = y.re * y.re * y.re;
            const double s3 = sum_cubes(y);
            vol += (double)texel_solid_angle(u0, u1, v0, v1) * ((double)re3 - s3 - chi_e * re3);
        }
        __syncthreads();   // the texels are reused
    }
    for (int off = 16; off > 0; off >>= 1) vol += __shfl_xor_sync(0xffffffffu, vol, off);
    if (lane == 0) part[warp] = vol;
    __syncthreads();
    if (tid == 0) {
        double tot = 0.0;
        for (int i = 0; i < kDirThreads / 32; ++i) tot += part[i];
        block_sum = tot;
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        double tot = 0.0;
        for (int g = 0; g < G; ++g) tot += *cluster.map_shared_rank(&block_sum, g);
        out[blockIdx.x / G] = tot / 3.0;   // once: a division a texel held a scheduler for 560 cycles
    }
    cluster.sync();   // no block leaves while its shared memory is read
}

}  // namespace

obb_status directional_outer_volume(obb_ctx* ctx, const obb_mesh* mesh, const obb_box* d_boxes, int64_t K, int32_t m,
                                    double* d_out)
{
    if (K <= 0) return OBB_OK;
    // Blocks per box: the fewest that put a block on every SM.  Each one
    // walks the whole mesh, so more only repeat that walk (64 boxes: three
    // blocks a box 0.066 ms, six 0.091 ms).
    const int64_t want = ctx->num_sms;
    const int G = K >= want ? 1 : 2 * K >= want ? 2 : 3 * K >= want ? 3 : 6;
    const int smem = (int)sizeof(DirTexel) * std::min(kDirTexels, 6 / G * m * m);
    OBB_CK(ctx, cudaFuncSetAttribute(k_directional, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(DirTexel) * kDirTexels));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(K * G));
    cfg.blockDim = dim3(kDirThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = ctx->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = G;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    OBB_CK(ctx, cudaLaunchKernelEx(&cfg, k_directional, (const float*)mesh->d_verts, (const int32_t*)mesh->d_tris,
                                   mesh->nt, d_boxes, m, (int32_t)G, d_out));
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

}  // namespace obbv
