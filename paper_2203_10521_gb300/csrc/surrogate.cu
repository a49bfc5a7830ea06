// Learned surrogate of the outer volume: a small MLP that predicts the empty
// fraction of a box from its parameters and an 8^3 occupancy patch sampled in
// the box's own frame.  The partition rounds of the Lloyd step use it to keep
// only the most promising candidate moves per cluster; the exact lattice count
// still decides every accepted move.
//
// Features (524 per box), from the quantised box alone, exact integers and
// then FP32 with a fixed operation order (so the patch bits are reproducible):
//   Lq, Hq = ceil(lo / 256), floor(hi / 256); M = n (3x3), M^-1 by cofactors;
//   sample s in {0..7}^3: v_a = Lq_a + (Hq_a - Lq_a) (2 s_a + 1) / 16,
//   p = M^-1 v, index = floor(p + 1/2), bit = occupancy (0 outside [0, N)^3);
//   box parameters: centre M^-1 (Lq + Hq) / 2 / N, axes n_0 / |n_0|, n_1 / |n_1|,
//   half widths (Hq_a - Lq_a) / (2 |n_a|) / N.
// Network: 524 -> 128 -> 128 -> 128 -> 1, ReLU, sigmoid output (the empty
// fraction); predicted outer volume = fraction x box volume in lattice cells
// (prod (Hq_a - Lq_a + 1) / |det M|).  Training: mean squared error on the
// fraction, Adam, FP32 master weights; inference reads an FP16 copy of the
// weights and accumulates in FP32 on the tensor cores; training and FP32
// inference keep FP32 products on CUDA cores.
#include <cuda_fp16.h>

#include <cmath>
#include <random>
#include <vector>

#include "internal.h"

namespace obbv {
namespace {

constexpr int kIn = kSurrogateInputs;
constexpr int kH = 128;

// parameter offsets in the flat vector: W1 b1 W2 b2 W3 b3 W4 b4 (W row-major [in][out])
constexpr int64_t oW1 = 0, oB1 = oW1 + (int64_t)kIn * kH, oW2 = oB1 + kH, oB2 = oW2 + kH * kH, oW3 = oB2 + kH,
                  oB3 = oW3 + kH * kH, oW4 = oB3 + kH, oB4 = oW4 + kH, kParams = oB4 + 1;

// ---------------------------------------------------------------- features

// What the samples of a box need: its centre and edges in index space, and its
// 12 parameters.
struct FeatureBox {
    float c[3], E[9], par[12];
};

// Per box, once: the exact adjugate A of the normals (n^-1 = A / det) in
// int64 and det in 128 bits, then FP32 with one rounding per operation in
// a fixed order (explicit _rn intrinsics: nothing is fused).  Integers
// reach FP32 as two 32-bit halves joined by one fmaf.
__device__ __forceinline__ void feature_box(const obb_qbox& q, int32_t N, FeatureBox* __restrict__ out)
{
    int64_t m[9], L[3], H[3];
    for (int i = 0; i < 9; ++i) m[i] = q.n[i];
    for (int a = 0; a < 3; ++a) {
        L[a] = -((-q.b[2 * a]) >> kS);
        H[a] = q.b[2 * a + 1] >> kS;
    }
    const int64_t A[9] = {m[4] * m[8] - m[5] * m[7], m[2] * m[7] - m[1] * m[8], m[1] * m[5] - m[2] * m[4],
                          m[5] * m[6] - m[3] * m[8], m[0] * m[8] - m[2] * m[6], m[2] * m[3] - m[0] * m[5],
                          m[3] * m[7] - m[4] * m[6], m[1] * m[6] - m[0] * m[7], m[0] * m[4] - m[1] * m[3]};
    const __int128 det = (__int128)m[0] * A[0] + (__int128)m[1] * A[3] + (__int128)m[2] * A[6];
    const float detf = i128_to_float(det);
    float Af[9], Sf[3], Df[3];
    for (int i = 0; i < 9; ++i) Af[i] = i64_to_float(A[i]);
    for (int a = 0; a < 3; ++a) {
        Sf[a] = i64_to_float(L[a] + H[a]);
        Df[a] = i64_to_float(H[a] - L[a]);
    }
    for (int r = 0; r < 3; ++r) {
        float c = 0.0f;
        if (det != 0) {
            // index-space centre: ((A_r0 S_0 + A_r1 S_1) + A_r2 S_2) / (2 det)
            const float t = __fadd_rn(__fadd_rn(__fmul_rn(Af[3 * r], Sf[0]), __fmul_rn(Af[3 * r + 1], Sf[1])),
                                      __fmul_rn(Af[3 * r + 2], Sf[2]));
            c = __fdiv_rn(t, __fmul_rn(2.0f, detf));
        }
        out->c[r] = c;
        out->par[r] = __fdiv_rn(c, (float)N);
        // edge a of the box in index space: (A_ra D_a) / det
        for (int a = 0; a < 3; ++a)
            out->E[3 * r + a] = det != 0 ? __fdiv_rn(__fmul_rn(Af[3 * r + a], Df[a]), detf) : 0.0f;
    }
    for (int a = 0; a < 3; ++a) {
        const float n0 = (float)q.n[3 * a], n1 = (float)q.n[3 * a + 1], n2 = (float)q.n[3 * a + 2];
        const float nn = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(n0, n0), __fmul_rn(n1, n1)), __fmul_rn(n2, n2)));
        if (a < 2) {
            out->par[3 + 3 * a] = nn > 0.0f ? __fdiv_rn(n0, nn) : 0.0f;
            out->par[4 + 3 * a] = nn > 0.0f ? __fdiv_rn(n1, nn) : 0.0f;
            out->par[5 + 3 * a] = nn > 0.0f ? __fdiv_rn(n2, nn) : 0.0f;
        }
        out->par[9 + a] = nn > 0.0f ? __fdiv_rn(__fdiv_rn(__fmul_rn(Df[a], 0.5f), nn), (float)N) : 0.0f;
    }
}

// 32 boxes a block (kFeatFew: eight): its first warp sets them up, a box a lane;
// then every warp samples four of them (one).  Patch point s is the centre plus the edges times
// g_a = (2 s_a - 7) / 16, ((c_r + E_r0 g_0) + E_r1 g_1) + E_r2 g_2, rounded to
// the nearest lattice point (floor(p + 1/2)); the bit is 0 outside the
// lattice.  A lane keeps s_0 and half of s_1, so of a sample's three sums only
// the last terms are left.  The bits come from the counting copy, whose
// neighbouring columns share a line.  A block per box, one thread setting it
// up, took 94.3 us for 32,768 boxes at 512^3; this takes 26.5 (41.1 with a
// branch around every load; batches of 1, 2 and 8 s_2: 26.4, 26.2, 27.4),
// 2.6 TB/s of written features.  While blocks of eight boxes all fit the
// machine at once, a warp has one box to sample instead of four in a row (300
// boxes 10.4 -> 6.4 us, 8.4 with a block per box; 3,000 10.5 -> 10.4).
constexpr int kFeatBoxes = 32, kFeatFew = 8;
constexpr int kFeatThreads = 256;
constexpr int kFeatBatch = 4;    // s_2 whose words a lane loads together
constexpr float kFloorMagic = 12582912.0f;         // 1.5 2^23: q + it, rounded down, ends with floor(q) for |q| < 2^22
constexpr uint32_t kFloorBits = 0x4b400000u;       // its bits

template <int kBoxes>
__global__ void __launch_bounds__(kFeatThreads) k_features(const obb_qbox* __restrict__ boxes,
                                                           const int32_t* __restrict__ d_K, int32_t K,
                                                           const uint64_t* __restrict__ cwords, int32_t N, int32_t W,
                                                           float* __restrict__ feats)
{
    __shared__ FeatureBox sh[kBoxes];
    if (d_K) K = *d_K;
    const int64_t k0 = blockIdx.x * (int64_t)kBoxes;
    if (k0 >= K) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp == 0 && lane < kBoxes && k0 + lane < K) {
        const obb_qbox q = boxes[k0 + lane];
        feature_box(q, N, &sh[lane]);
    }
    __syncthreads();
    const float g0 = __fmul_rn((float)(2 * (lane & 7) - 7), 0.0625f);
    const float g1[2] = {__fmul_rn((float)(2 * (lane >> 3) - 7), 0.0625f),
                         __fmul_rn((float)(2 * (4 + (lane >> 3)) - 7), 0.0625f)};
    for (int i = warp; i < kBoxes && k0 + i < K; i += kFeatThreads / 32) {
        const FeatureBox& b = sh[i];
        float* f = feats + (k0 + i) * (int64_t)kIn;
        if (lane < 12) f[lane] = b.par[lane];
        float t[2][3];   // (c_r + E_r0 g_0) + E_r1 g_1 for the lane's two s_1
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float u = __fadd_rn(b.c[r], __fmul_rn(b.E[3 * r], g0));
            t[0][r] = __fadd_rn(u, __fmul_rn(b.E[3 * r + 1], g1[0]));
            t[1][r] = __fadd_rn(u, __fmul_rn(b.E[3 * r + 1], g1[1]));
        }
        const uint32_t* w32 = reinterpret_cast<const uint32_t*>(cwords);
#pragma unroll
        for (int s4 = 0; s4 < 8; s4 += kFeatBatch) {
            // the batch's words are all loaded before the first is used; a sample outside the lattice reads word 0
            uint32_t word[2 * kFeatBatch], sh_bit[2 * kFeatBatch];
#pragma unroll
            for (int u = 0; u < 2 * kFeatBatch; ++u) {
                const int s2 = s4 + u / 2, h = u & 1;
                const float g2 = (float)(2 * s2 - 7) * 0.0625f;
                // floor(p + 1/2) from the bits of a sum rounded down; any value outside [0, N), infinities and
                // NaN included, compares above N as an unsigned number
                uint32_t x[3];
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    x[r] = __float_as_uint(__fadd_rd(__fadd_rn(__fadd_rn(t[h][r], __fmul_rn(b.E[3 * r + 2], g2)), 0.5f),
                                                     kFloorMagic)) - kFloorBits;
                const bool in = max(x[0], max(x[1], x[2])) < (uint32_t)N;
                const uint32_t at = 2u * ((x[2] * (uint32_t)W + (x[0] >> 6)) * (uint32_t)N + x[1]) + (x[0] >> 5 & 1u);
                word[u] = __ldg(w32 + (in ? at : 0u));   // at most 2048^2 64 32-bit words
                sh_bit[u] = in ? x[0] & 31u : 32u;
            }
#pragma unroll
            for (int u = 0; u < 2 * kFeatBatch; ++u)
                f[12 + 64 * (s4 + u / 2) + 32 * (u & 1) + lane] =
                    (uint64_t)word[u] >> sh_bit[u] & 1u ? 1.0f : 0.0f;
        }
    }
}

static void launch_features(obb_ctx* ctx, const obb_lattice* lat, const obb_qbox* boxes, const int32_t* d_K, int64_t K,
                            float* feats)
{
    const auto run = [&](auto kernel, int per) {
        kernel<<<(unsigned)((K + per - 1) / per), kFeatThreads, 0, ctx->stream>>>(boxes, d_K, (int32_t)K, lat->d_cwords,
                                                                                  lat->frame.N, lat->frame.W, feats);
    };
    if (K <= 4 * kFeatFew * (int64_t)ctx->num_sms) run(k_features<kFeatFew>, kFeatFew);
    else run(k_features<kFeatBoxes>, kFeatBoxes);
    note_launch(ctx);
}

// ------------------------------------------------------ tensor-core forward
//
// Inference of the screening network on the 5th-generation tensor cores: one
// CTA (4 warps) carries 128 boxes through all four layers.  Operands are FP16
// in shared memory in the canonical K-major layout without swizzle (8 x 8
// "core matrices" of 128 contiguous bytes: core (r / 8, c / 8) of a tile with
// C columns at ((r / 8) (C / 8) + c / 8) * 128 bytes, so the leading (K)
// byte offset is 128 and the stride (M/N) byte offset C * 16).  One thread
// issues tcgen05.mma (kind::f16, M = N = 128, K = 16 per instruction, FP32
// accumulator in 128 TMEM columns) and commits to an mbarrier; every thread
// then reads its own row of the accumulator (TMEM lane = box) with
// tcgen05.ld, adds the bias, applies ReLU and writes FP16 back as the next
// layer's A operand.  The 128 -> 1 output layer is a dot product per row in
// registers.  Every wait is bounded; a CTA that allocated TMEM frees it on
// every path.

constexpr int kTcRows = 128;                    // boxes per CTA (= TMEM lanes)
constexpr int kTcK1 = 576;                      // layer-1 K (524 features) padded to chunks of 64
constexpr int kTcChunk = 64;                    // layer-1 K per staged chunk
constexpr uint32_t kTcCols = 128;               // TMEM columns (one FP32 accumulator)
// instruction descriptor: D = FP32 (bits 4-5), A = B = FP16 (bits 7-12 zero),
// both K-major (bits 15, 16 zero), N / 8 at bits 17-22, M / 16 at bits 24-28
constexpr uint32_t kTcIdesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
constexpr uint64_t kTcWaitNs = 250000000ull;    // a wait gives up after 250 ms (device global timer)

__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start, leading and stride byte offsets
// (>> 4), descriptor version 1 (bits 46-47), no swizzle (bits 61-63 = 0)
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3fffu) | ((uint64_t)((lbo >> 4) & 0x3fffu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3fffu) << 32) | (1ull << 46);
}

// byte offset of element (r, c) in a K-major no-swizzle tile of C columns
__device__ __forceinline__ uint32_t tc_off(int r, int c, int C)
{
    return (uint32_t)((((r >> 3) * (C >> 3) + (c >> 3)) << 7) + ((r & 7) << 4) + ((c & 7) << 1));
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(kTcIdesc), "r"(accumulate));
}

__device__ __forceinline__ void tc_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// wait for the given phase of the mbarrier; false once kTcWaitNs have passed
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t phase)
{
    const uint64_t t0 = global_ns();
    for (;;) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(smem_addr(bar)), "r"(phase)
            : "memory");
        if (ok) return true;
        if (global_ns() - t0 > kTcWaitNs) return false;
    }
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float* v)
{
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic-proxy shared-memory writes made visible to the tensor core (async proxy)
__device__ __forceinline__ void tc_fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }


// bulk copy (TMA, untiled) of `bytes` from global to shared memory, completing
// on `bar` (16-byte aligned addresses, a multiple of 16 bytes)
__device__ __forceinline__ void tc_bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile(
        "{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}\n" ::"r"(smem_addr(bar)),
        "r"(bytes)
        : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// FP16 weights, transposed (N x K, K-major) and laid out as the kernel's shared
// tiles: W1 as 9 chunks of 128 x 64 (K zero-padded to 576), then W2, W3 as
// 128 x 128 tiles
constexpr int64_t kTcW1Chunk = (int64_t)kH * kTcChunk;               // halves per W1 chunk
constexpr int64_t kTcPacked = (kTcK1 / kTcChunk) * kTcW1Chunk + 2 * (int64_t)kH * kH;

// shared memory: two layer-1 A chunks, later h (32 KB); two W1 chunks, later
// W3 (32 KB); W2 (32 KB); biases, w4, b4.  Two CTAs on an SM hold 32,768 boxes
// in one wave.
constexpr int kTcSmem = 3 * 32768 + (4 * kH + 4) * 4;

// y = sigmoid(W4 relu(W3 relu(W2 relu(W1 x + b1) + b2) + b3) + b4) for rows
// [128 blockIdx.x, +128) of X (the live row count is *d_M when given).
// Layer 1 reads 2 KB of features a box and bounds the kernel: its nine chunks
// are pipelined (a chunk's features are loaded into registers, sixteen bytes
// a load, while the tensor core works on the chunk before; W1 chunks arrive
// one ahead), and W2 and W3 arrive under earlier layers.  One chunk after
// another, with four-byte loads: 38.6 us for 32,768 boxes; this way 25.6.
__global__ void __launch_bounds__(kTcRows) k_mlp_tc(const float* __restrict__ X, int M, const int32_t* __restrict__ d_M,
                                                    const __half* __restrict__ wtc, const __half* __restrict__ wh,
                                                    const float* __restrict__ w, float* __restrict__ y,
                                                    int32_t* __restrict__ err, int32_t stall)
{
    // stall (test hook): the first MMA group is neither issued nor committed,
    // so its wait can only give up; nothing of it is left in flight
    if (d_M) M = min(M, *d_M);
    const int m0 = blockIdx.x * kTcRows;
    if (m0 >= M) return;   // uniform: the whole CTA leaves before any TMEM or barrier use
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    unsigned char* sA = tc_smem;            // A operand: layer-1 chunks (128 x 64, two), then h (128 x 128)
    unsigned char* sB = tc_smem + 32768;    // B operand: W1 chunks (two), then W3
    unsigned char* sC = tc_smem + 65536;    // B operand: W2
    float* sBias = reinterpret_cast<float*>(tc_smem + 3 * 32768);   // b1, b2, b3, w4 (4 x 128), b4
    __shared__ __align__(8) uint64_t bar_mma, bar_ld[2], bar_w;
    __shared__ uint32_t s_tmem;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    constexpr int kChunks = kTcK1 / kTcChunk;
    constexpr int kHalf = 16384;            // bytes of a layer-1 chunk of A or B

    // A warp's 32 rows x 64 columns of a chunk: eight pieces of eight
    // columns a thread, 8 rows x 4 pieces a step (128 bytes of a row from
    // global memory, conflict-free 16-byte stores to the operand tile)
    const bool wide = (reinterpret_cast<uintptr_t>(X) & 15) == 0;   // rows are multiples of 16 bytes
    float4 x[8][2];
    auto load_x = [&](int q) {
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const int m = m0 + 32 * warp + 8 * (n >> 1) + (lane & 7), k = kTcChunk * q + 8 * (4 * (n & 1) + (lane >> 3));
            const float* p = X + (int64_t)m * kIn + k;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (m < M && k + 4 * h < kIn) {   // kIn is a multiple of 4
                    if (wide) v = __ldg(reinterpret_cast<const float4*>(p + 4 * h));
                    else v = make_float4(__ldg(p + 4 * h), __ldg(p + 4 * h + 1), __ldg(p + 4 * h + 2), __ldg(p + 4 * h + 3));
                }
                x[n][h] = v;
            }
        }
    };
    auto store_x = [&](unsigned char* dst) {
#pragma unroll
        for (int n = 0; n < 8; ++n) {
            const int r = 32 * warp + 8 * (n >> 1) + (lane & 7), c = 8 * (4 * (n & 1) + (lane >> 3));
            __align__(16) __half hv[8] = {__float2half_rn(x[n][0].x), __float2half_rn(x[n][0].y),
                                          __float2half_rn(x[n][0].z), __float2half_rn(x[n][0].w),
                                          __float2half_rn(x[n][1].x), __float2half_rn(x[n][1].y),
                                          __float2half_rn(x[n][1].z), __float2half_rn(x[n][1].w)};
            *reinterpret_cast<uint4*>(dst + tc_off(r, c, kTcChunk)) = *reinterpret_cast<const uint4*>(hv);
        }
    };
    load_x(0);

    for (int i = t; i < kH; i += kTcRows) {
        sBias[i] = w[oB1 + i];
        sBias[kH + i] = w[oB2 + i];
        sBias[2 * kH + i] = w[oB3 + i];
        sBias[3 * kH + i] = __half2float(wh[oW4 + i]);
    }
    if (t == 0) {
        sBias[4 * kH] = w[oB4];
        uint64_t* bars[4] = {&bar_mma, &bar_ld[0], &bar_ld[1], &bar_w};
        for (uint64_t* b : bars) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(b)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                     "r"(kTcCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t aS = smem_addr(sA), bS = smem_addr(sB), cS = smem_addr(sC);
    const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);   // this warp's 32 TMEM lanes
    const __half* w2 = wtc + kChunks * kTcW1Chunk;
    uint32_t mma = 0;           // groups committed, the same in every thread
    uint32_t loads = 1;         // thread 0: copies of W1 chunks and W3 issued, in turn on bar_ld[0] and bar_ld[1]
    bool ok = true;
    if (t == 0) {
        tc_bulk_load(sB, wtc, (uint32_t)(kTcW1Chunk * 2), &bar_ld[0]);
        tc_bulk_load(sC, w2, (uint32_t)(kH * kH * 2), &bar_w);
    }

    // Layer 1, chunk q: its features into A half q & 1 (free: the MMAs of
    // chunk q - 2 were waited for), the next features on their way, W1 chunk
    // q + 1 into the half that the MMAs of chunk q - 1 have left, then the
    // MMAs of chunk q.
    for (int q = 0; q < kChunks && ok; ++q) {
        const int half = q & 1;
        store_x(sA + half * kHalf);
        tc_fence_smem();
        if (q + 1 < kChunks) load_x(q + 1);
        bool got = true;
        if (q > 0) got = tc_wait(&bar_mma, (mma - 1) & 1);   // the MMAs of chunk q - 1
        if (q + 1 < kChunks && t == 0 && got) {
            tc_bulk_load(sB + (half ^ 1) * kHalf, wtc + (q + 1) * kTcW1Chunk, (uint32_t)(kTcW1Chunk * 2),
                         &bar_ld[half ^ 1]);
            ++loads;
        }
        got = got && tc_wait(&bar_ld[half], (q >> 1) & 1);
        tc_fence_before();
        ok = __syncthreads_and(got);
        if (!ok) break;
        if (t == 0 && !(stall && q == 0)) {
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < kTcChunk / 16; ++j)
                tc_mma(tmem, tc_desc(aS + half * kHalf + 256 * j, 128, kTcChunk * 16),
                       tc_desc(bS + half * kHalf + 256 * j, 128, kTcChunk * 16), (q > 0 || j > 0) ? 1u : 0u);
            tc_commit(&bar_mma);
        }
        ++mma;
    }
    if (ok) ok = __syncthreads_and(tc_wait(&bar_mma, (mma - 1) & 1));

    // layers 2 and 3: the accumulator row of this thread (TMEM lane = row)
    // becomes FP16 h in the A tile; W2 is there, W3 arrives meanwhile in the
    // place of the W1 chunks
    for (int layer = 0; layer < 2 && ok; ++layer) {
        if (layer == 0 && t == 0) {
            tc_bulk_load(sB, w2 + kH * kH, (uint32_t)(kH * kH * 2), &bar_ld[kChunks & 1]);
            ++loads;
        }
        tc_fence_after();
        for (int c = 0; c < kH / 32; ++c) {
            float v[32];
            tc_ld32(lane_base + 32 * c, v);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                __align__(16) __half hv[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) hv[e] = __float2half_rn(fmaxf(v[8 * g + e] + sBias[layer * kH + 32 * c + 8 * g + e], 0.f));
                *reinterpret_cast<uint4*>(sA + tc_off(t, 32 * c + 8 * g, kH)) = *reinterpret_cast<const uint4*>(hv);
            }
        }
        tc_fence_smem();
        const bool got = layer == 0 ? tc_wait(&bar_w, 0) : tc_wait(&bar_ld[kChunks & 1], (kChunks >> 1) & 1);
        tc_fence_before();
        ok = __syncthreads_and(got);
        if (!ok) break;
        if (t == 0) {
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < kH / 16; ++j)
                tc_mma(tmem, tc_desc(aS + 256 * j, 128, kH * 16), tc_desc((layer == 0 ? cS : bS) + 256 * j, 128, kH * 16),
                       j > 0 ? 1u : 0u);
            tc_commit(&bar_mma);
        }
        ++mma;
        ok = __syncthreads_and(tc_wait(&bar_mma, (mma - 1) & 1));
    }

    if (ok) {
        // output layer: relu(h3) . w4 + b4 per row, then the sigmoid
        tc_fence_after();
        float acc = sBias[4 * kH];
        for (int c = 0; c < kH / 32; ++c) {
            float v[32];
            tc_ld32(lane_base + 32 * c, v);
#pragma unroll
            for (int e = 0; e < 32; ++e)
                acc = fmaf(fmaxf(v[e] + sBias[2 * kH + 32 * c + e], 0.f), sBias[3 * kH + 32 * c + e], acc);
        }
        const int m = m0 + t;
        if (m < M) y[m] = 1.f / (1.f + __expf(-acc));
    } else {
        // a wait gave up: thread 0, which issued everything, reports it and
        // lets its tensor-core work and copies in flight finish (bounded);
        // TMEM is freed below
        if (t == 0) {
            atomicOr(err, kErrTimeout);
            if (mma > 0 && !stall) tc_wait(&bar_mma, (mma - 1) & 1);
            for (uint32_t i = loads > 1 ? loads - 2 : 0; i < loads; ++i) tc_wait(&bar_ld[i & 1], (i >> 1) & 1);
            tc_wait(&bar_w, 0);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols));
}

// box volume in lattice cells: prod (Hq_a - Lq_a + 1) / |det n|
__device__ __forceinline__ float box_cells(const obb_qbox& q)
{
    double M[9];
    for (int i = 0; i < 9; ++i) M[i] = (double)q.n[i];
    const double det = M[0] * (M[4] * M[8] - M[5] * M[7]) + M[1] * (M[5] * M[6] - M[3] * M[8]) +
                       M[2] * (M[3] * M[7] - M[4] * M[6]);
    double v = 1.0;
    for (int a = 0; a < 3; ++a) {
        const double w = (double)((q.b[2 * a + 1] >> kS) - (-((-q.b[2 * a]) >> kS)) + 1);
        v *= w > 0.0 ? w : 0.0;
    }
    return det != 0.0 ? (float)(v / fabs(det)) : 0.f;
}

// ------------------------------------------------------- FP32 network
//
// Training and FP32 inference run on CUDA cores in FP32 (no reduced-precision
// products).  An Adam step is three kernels:
//   k_mlp_rows   forward and backward of R rows a block: activations stay in
//                shared memory, the weights stream through a ring;
//   k_mlp_wgrad  all weight and bias gradients;
//   k_adam       the update, and every copy of the weights that a kernel
//                reads.
// Every sum is one chain of fused multiply-adds in ascending order (inputs of
// a neuron, rows of a batch): training amplifies any rounding (a sign of a
// pre-activation near zero), and a fixed order keeps a run reproducible
// whatever the tiles are.  A layer at a time as 64 x 64 tiles the step was 18
// launches, most of 2 to 32 blocks (0.83 ms at a batch of 1,024); the three
// kernels take 0.043 ms (23.9 + 15.7 + 2.9 us).

constexpr int kRowsThreads = kH;   // a thread per column
constexpr int kRowsBatch = 32;     // weight rows a thread loads ahead
constexpr int kIn4 = kIn / 4;
static_assert(kIn % 4 == 0, "features are read four at a time");

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int n>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(n) : "memory");
}

// bytes of k_mlp_rows' dynamic shared memory: features and activations
// [k][R], and the rows past the last that its read-ahead touches
constexpr int rows_smem(int R, bool train)
{
    return (int)sizeof(float) * (kIn * R + (train ? 4 : 2) * kH * R + 32);
}

struct RowsOut {   // training only: [B][128] activations and gradients, [B] output gradients, loss per block
    float *h1, *h2, *h3, *d1, *d2, *d3, *dy, *loss;
};

// Rows [R blockIdx.x, + R) of X through the network; y = the predicted
// fractions.  kTrain: also the gradients of the mean squared error against
// target down to the first layer's pre-activations.  A thread owns a column
// and R rows, so it alone needs its column's weights: it loads them (the
// transposed copies in wt on the way back) straight into registers, 32 rows
// ahead and across the layers, and each serves R products; the inputs are
// broadcast reads of shared memory, read four products' groups ahead.
// Staging the weights in shared memory by cp.async instead costs its writes
// and a barrier per chunk: 25.7 against 23.9 us at a batch of 1,024 (64 rows
// ahead: 26.3 us).
// R = 8 puts that batch on 128 SMs, a warp per scheduler, so the loop lives
// on instruction-level parallelism; R = 16 halves the passes over the weights
// (0.4 MB a block, from L2) once there are blocks enough.
template <int R, bool kTrain>
__global__ void __launch_bounds__(kRowsThreads) k_mlp_rows(const float* __restrict__ X, int M,
                                                           const int32_t* __restrict__ d_M,
                                                           const float* __restrict__ w, const float* __restrict__ wt,
                                                           const float* __restrict__ target, float* __restrict__ y,
                                                           RowsOut out)
{
    if (d_M) M = min(M, *d_M);
    const int m0 = blockIdx.x * R;
    if (m0 >= M) return;   // uniform
    extern __shared__ __align__(16) float rows_smem_base[];
    float* xs = rows_smem_base;
    float* act = xs + kIn * R;                              // [2 or 4][kH][R]
    __shared__ float s_dy[R], s_l[R], s_w4[kH];
    const int tid = threadIdx.x;

    // what the ends of the layers need, loaded up front
    const float bias1 = __ldg(w + oB1 + tid), bias2 = __ldg(w + oB2 + tid), bias3 = __ldg(w + oB3 + tid),
                w4 = __ldg(w + oW4 + tid), b4 = __ldg(w + oB4);
    const float want = kTrain && tid < R && m0 + tid < M ? __ldg(target + m0 + tid) : 0.f;
    float cur[kRowsBatch], nxt[kRowsBatch];   // this column's weights: the batch in use, the one after it
    auto load = [&](float (&v)[kRowsBatch], const float* src, int rows) {
#pragma unroll
        for (int i = 0; i < kRowsBatch; ++i) v[i] = i < rows ? __ldg(src + i * kH) : 0.f;
    };
    load(cur, w + oW1 + tid, kRowsBatch);
    s_w4[tid] = w4;

    // the features, transposed to [k][R]; rows past M are zero
    if ((reinterpret_cast<uintptr_t>(X) & 15) == 0) {
        for (int i = tid; i < R * kIn4; i += kRowsThreads) {
            const int r = i / kIn4, k = 4 * (i % kIn4);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (m0 + r < M) v = __ldg(reinterpret_cast<const float4*>(X + (int64_t)(m0 + r) * kIn + k));
            xs[k * R + r] = v.x;
            xs[(k + 1) * R + r] = v.y;
            xs[(k + 2) * R + r] = v.z;
            xs[(k + 3) * R + r] = v.w;
        }
    } else {
        for (int i = tid; i < R * kIn; i += kRowsThreads) {
            const int r = i / kIn, k = i % kIn;
            xs[k * R + r] = m0 + r < M ? __ldg(X + (int64_t)(m0 + r) * kIn + k) : 0.f;
        }
    }

    float acc[R];
    // acc[r] = sum over k of in[k][r] times weight row k of this column (wp); next: the weights after these.
    // The barrier orders what was written to `in` before, and the readers of the buffer written after.
    auto layer = [&](const float* in, int K, const float* wp, const float* next) {
        constexpr int G = 32 / R;   // inputs read together: 32 floats
        __syncthreads();
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = 0.f;
        for (int k0 = 0; k0 < K; k0 += kRowsBatch) {
            const int rows = min(kRowsBatch, K - k0), after = K - k0 - kRowsBatch;
            if (after > 0) load(nxt, wp + (k0 + kRowsBatch) * kH, after);
            else if (next) load(nxt, next, kRowsBatch);
            float4 x[2][8];
            auto read = [&](float4 (&v)[8], int k) {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = *reinterpret_cast<const float4*>(in + k * R + 4 * i);
            };
            read(x[0], k0);
#pragma unroll
            for (int g = 0; g < kRowsBatch / G; ++g) {
                if (g * G >= rows) break;   // K is a multiple of 4
                if (g + 1 < kRowsBatch / G) read(x[(g + 1) & 1], k0 + (g + 1) * G);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 v = x[g & 1][i];
                    const float wv = cur[g * G + 4 * i / R];
                    const int r = 4 * i % R;
                    acc[r] = fmaf(v.x, wv, acc[r]);
                    acc[r + 1] = fmaf(v.y, wv, acc[r + 1]);
                    acc[r + 2] = fmaf(v.z, wv, acc[r + 2]);
                    acc[r + 3] = fmaf(v.w, wv, acc[r + 3]);
                }
            }
#pragma unroll
            for (int i = 0; i < kRowsBatch; ++i) cur[i] = nxt[i];
        }
    };
    // acc to an activation buffer [column][R] and, in training, to [B][128]
    auto store = [&](float* a, float* h) {
        if (a)
#pragma unroll
            for (int r = 0; r < R; r += 4)
                *reinterpret_cast<float4*>(a + tid * R + r) = make_float4(acc[r], acc[r + 1], acc[r + 2], acc[r + 3]);
        if (kTrain)
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (m0 + r < M) h[(int64_t)(m0 + r) * kH + tid] = acc[r];
    };
    float* a1 = act;
    float* a2 = act + kH * R;
    float* a3 = kTrain ? act + 2 * kH * R : a1;
    float* da = act + 3 * kH * R;
    // a gradient passes where its activation is positive
    auto masked = [&](const float* a) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (!(a[tid * R + r] > 0.f)) acc[r] = 0.f;
    };
    // one copy of the loop's code for the three layers and the two steps back (five copies do not fit the
    // instruction caches)
#pragma unroll 1
    for (int l = 0; l < (kTrain ? 5 : 3); ++l) {
        const float *w2 = w + oW2 + tid, *w3 = w + oW3 + tid, *w3t = wt + kH * kH + tid, *w2t = wt + tid;
        layer(l == 0 ? xs : l == 1 ? a1 : l == 2 ? a2 : l == 3 ? da : a3, l == 0 ? kIn : kH,
              l == 0 ? w + oW1 + tid : l == 1 ? w2 : l == 2 ? w3 : l == 3 ? w3t : w2t,
              l == 0 ? w2 : l == 1 ? w3 : l == 2 ? (kTrain ? w3t : nullptr) : l == 3 ? w2t : nullptr);
        if (l < 3) {
            const float bias = l == 0 ? bias1 : l == 1 ? bias2 : bias3;
#pragma unroll
            for (int r = 0; r < R; ++r) acc[r] = fmaxf(acc[r] + bias, 0.f);
            store(l == 0 ? a1 : l == 1 ? a2 : a3, l == 0 ? out.h1 : l == 1 ? out.h2 : out.h3);
        } else if (l == 3) {
            masked(a2);
            store(a3, out.d2);
        } else {
            masked(a1);
            store(nullptr, out.d1);
        }
        if (l != 2) continue;
        __syncthreads();
        // the output neuron: a thread per row
        if (tid < R) {
            float v = 0.f;
#pragma unroll 16
            for (int k = 0; k < kH; ++k) v = fmaf(a3[k * R + tid], s_w4[k], v);
            const int m = m0 + tid;
            const float f = 1.f / (1.f + __expf(-(v + b4)));
            if (m < M) y[m] = f;
            if (kTrain) {
                const float e = m < M ? f - want : 0.f;
                s_dy[tid] = 2.f * e / (float)M * f * (1.f - f);
                s_l[tid] = e * e / (float)M;
                if (m < M) out.dy[m] = s_dy[tid];
            }
        }
        if (!kTrain) return;
        __syncthreads();
        if (tid == 0) {
            float l = 0.f;
            for (int r = 0; r < R; ++r) l += s_l[r];
            out.loss[blockIdx.x] = l;
        }
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = s_dy[r] * w4;
        masked(a3);
        store(da, out.d3);
    }
}

// Weight and bias gradients, one block a piece of them:
//   block 0               the output neuron's bias (sum of dy);
//   blocks 1-8            its weights, 16 inputs each;
//   blocks 9-20           the other biases, 32 columns each: sums of 256
//                         strided chains as a tree of shuffles would add them;
//   the rest              16 x 16 tiles of A^T D (A = a layer's inputs, D =
//                         the gradients of its pre-activations).
// A weight's chain runs over the whole batch, so the parallelism is across
// weights: 392 tiles of two warps, a thread holding 2 x 2 sums (16 x 32 tiles
// of two warps: 19.6, of four: 17.1 against 15.7 us: fewer blocks than two
// an SM leave some with one, and 2 x 4 sums leave a warp's issue the limit).
// Both operands are read along their rows, so nothing is
// transposed; 64-row stages arrive by cp.async three ahead.
constexpr int kGradThreads = 64;
constexpr int kGradM = 16, kGradN = 16;
constexpr int kGradRows = 64;      // batch rows per stage
constexpr int kGradStages = 4;
constexpr int kGradNt = kH / kGradN;
constexpr int kGradTiles1 = (kIn + kGradM - 1) / kGradM * kGradNt, kGradTilesH = kH / kGradM * kGradNt;
constexpr int kGradBlocks = 21 + kGradTiles1 + 2 * kGradTilesH;
constexpr int kGradStage = kGradRows * (kGradM + kGradN);          // floats
constexpr int kGradSmem = (int)sizeof(float) * kGradStages * kGradStage;
static_assert(kGradRows * 17 <= kGradStage, "16 inputs and dy fit a stage");

__global__ void __launch_bounds__(kGradThreads) k_mlp_wgrad(const float* __restrict__ X, int M, const RowsOut in,
                                                            float* __restrict__ grad)
{
    extern __shared__ __align__(16) float grad_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int steps = (M + kGradRows - 1) / kGradRows;
    if (blockIdx.x == 0) {
        for (int q = warp; q < 8; q += 2) {
            float s = 0.f;
            for (int m = 32 * q + lane; m < M; m += 256) s += __ldg(in.dy + m);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) grad_smem[q] = s;
        }
        __syncthreads();
        if (tid == 0) {
            float t = 0.f;
            for (int q = 0; q < 8; ++q) t += grad_smem[q];
            grad[oB4] = t;
        }
        return;
    }
    if (blockIdx.x < 9) {
        const int i0 = 16 * (blockIdx.x - 1);
        auto issue = [&](int st) {
            if (st < steps) {
                float* a = grad_smem + (st % kGradStages) * kGradStage;
                const int b = st * kGradRows, rows = min(kGradRows, M - b);
                for (int i = tid; i < rows * 4; i += kGradThreads)
                    cp_async16(a + 4 * i, in.h3 + (int64_t)(b + i / 4) * kH + i0 + 4 * (i % 4));
                if (tid < rows) cp_async4(a + kGradRows * 16 + tid, in.dy + b + tid);
            }
            cp_commit();
        };
        for (int st = 0; st < kGradStages - 1; ++st) issue(st);
        float s = 0.f;
        for (int st = 0; st < steps; ++st) {
            cp_wait<kGradStages - 2>();
            __syncthreads();
            issue(st + kGradStages - 1);
            const float* a = grad_smem + (st % kGradStages) * kGradStage;
            const int rows = min(kGradRows, M - st * kGradRows);
            if (tid < 16)
#pragma unroll 16
                for (int r = 0; r < rows; ++r) s = fmaf(a[r * 16 + tid], a[kGradRows * 16 + r], s);
        }
        if (tid < 16) grad[oW4 + i0 + tid] = s;
        return;
    }
    if (blockIdx.x < 21) {
        const int l = (blockIdx.x - 9) / 4, n = 32 * ((blockIdx.x - 9) % 4) + lane;
        const float* D = l == 0 ? in.d1 : l == 1 ? in.d2 : in.d3;
        for (int q = warp; q < 8; q += 2) {
            float s[32];
#pragma unroll
            for (int v = 0; v < 32; ++v) s[v] = 0.f;
            for (int m = 32 * q; m < M; m += 256) {
                float x[32];
#pragma unroll
                for (int v = 0; v < 32; ++v) x[v] = m + v < M ? __ldg(D + (int64_t)(m + v) * kH + n) : 0.f;
#pragma unroll
                for (int v = 0; v < 32; ++v) s[v] += x[v];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int v = 0; v < o; ++v) s[v] += s[v + o];
            grad_smem[32 * q + lane] = s[0];
        }
        __syncthreads();
        if (warp == 0) {
            float t = 0.f;
            for (int q = 0; q < 8; ++q) t += grad_smem[32 * q + lane];
            grad[(l == 0 ? oB1 : l == 1 ? oB2 : oB3) + n] = t;
        }
        return;
    }
    int tile = blockIdx.x - 21, ld = kH;
    const float *A, *D;
    int64_t oW;
    if (tile < kGradTiles1) {
        A = X, D = in.d1, ld = kIn, oW = oW1;
    } else if ((tile -= kGradTiles1) < kGradTilesH) {
        A = in.h1, D = in.d2, oW = oW2;
    } else {
        tile -= kGradTilesH;
        A = in.h2, D = in.d3, oW = oW3;
    }
    const int m0 = tile / kGradNt * kGradM, n0 = tile % kGradNt * kGradN, width = min(kGradM, ld - m0);
    const bool wide = (reinterpret_cast<uintptr_t>(A) & 15) == 0;   // ld and m0 are multiples of 4
    // this thread's share of a stage: 4 of the 64 x 4 pieces of A and of D
    const int ar = tid >> 2, aq = 4 * (tid & 3);
    const float* asrc = A + (int64_t)ar * ld + m0 + aq;
    const float* dsrc = D + (int64_t)ar * kH + n0 + aq;
    auto issue = [&](int st) {
        if (st < steps) {
            float* a = grad_smem + (st % kGradStages) * kGradStage + ar * kGradM + aq;
            float* d = a + kGradRows * kGradM;
            const int b = st * kGradRows, rows = min(kGradRows, M - b);
            const float* as = asrc + (int64_t)b * ld;
            const float* ds = dsrc + (int64_t)b * kH;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (ar + 16 * i < rows) {
                    if (aq < width) {
                        if (wide) cp_async16(a + 16 * i * kGradM, as + 16 * i * ld);
                        else
                            for (int e = 0; e < 4; ++e) cp_async4(a + 16 * i * kGradM + e, as + 16 * i * ld + e);
                    }
                    cp_async16(d + 16 * i * kGradN, ds + 16 * i * kH);
                }
        }
        cp_commit();
    };
    for (int st = 0; st < kGradStages - 1; ++st) issue(st);
    // a warp covers 8 rows x 16 columns
    const int mr = 8 * warp + 2 * (lane >> 3), nc = 2 * (lane & 7);
    float acc[2][2] = {};
    for (int st = 0; st < steps; ++st) {
        cp_wait<kGradStages - 2>();
        __syncthreads();
        issue(st + kGradStages - 1);
        const float* a = grad_smem + (st % kGradStages) * kGradStage + mr;
        const float* d = grad_smem + (st % kGradStages) * kGradStage + kGradRows * kGradM + nc;
        auto rows8 = [&](int r0, int n) {   // n <= 8 rows, all reads before the products
            float2 av[8], dv[8];
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (r < n) {
                    av[r] = *reinterpret_cast<const float2*>(a + (r0 + r) * kGradM);
                    dv[r] = *reinterpret_cast<const float2*>(d + (r0 + r) * kGradN);
                }
#pragma unroll
            for (int r = 0; r < 8; ++r)
                if (r < n) {
                    acc[0][0] = fmaf(av[r].x, dv[r].x, acc[0][0]);
                    acc[0][1] = fmaf(av[r].x, dv[r].y, acc[0][1]);
                    acc[1][0] = fmaf(av[r].y, dv[r].x, acc[1][0]);
                    acc[1][1] = fmaf(av[r].y, dv[r].y, acc[1][1]);
                }
        };
        const int rows = min(kGradRows, M - st * kGradRows);
        if (rows == kGradRows) {
#pragma unroll
            for (int r = 0; r < kGradRows; r += 8) rows8(r, 8);
        } else {
            for (int r = 0; r < rows; r += 8) rows8(r, rows - r);
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)   // rows past `width` hold nothing that is used
        if (mr + i < width)
#pragma unroll
            for (int j = 0; j < 2; ++j) grad[oW + (int64_t)(m0 + mr + i) * kH + n0 + nc + j] = acc[i][j];
}

// the loss: the blocks' sums, by the first warp in a fixed order
__device__ __forceinline__ void sum_loss(const float* __restrict__ parts, int n, float* __restrict__ loss)
{
    if (blockIdx.x != 0 || threadIdx.x >= 32) return;
    float l = 0.f;
    for (int i = threadIdx.x; i < n; i += 32) l += parts[i];
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (threadIdx.x == 0) *loss = l;
}

__global__ void k_loss(const float* __restrict__ parts, int n, float* __restrict__ loss) { sum_loss(parts, n, loss); }

// the copies of weight i: FP16, its place in the tensor-core kernel's tiles,
// and W2, W3 transposed
__device__ __forceinline__ void store_weight_copies(int64_t i, float wi, __half* __restrict__ wh,
                                                    __half* __restrict__ wtc, float* __restrict__ wt)
{
    const __half h = __float2half_rn(wi);
    wh[i] = h;
    if (i < oB1) {
        const int n = (int)(i % kH), k = (int)(i / kH);
        wtc[(k / kTcChunk) * kTcW1Chunk + tc_off(n, k % kTcChunk, kTcChunk) / 2] = h;
    } else if ((i >= oW2 && i < oB2) || (i >= oW3 && i < oB3)) {
        const int layer = i >= oW3, j = (int)(i - (layer ? oW3 : oW2)), n = j % kH, k = j / kH;
        wtc[(kTcK1 / kTcChunk) * kTcW1Chunk + layer * kH * kH + tc_off(n, k, kH) / 2] = h;
        wt[layer * kH * kH + n * kH + k] = wi;
    }
}

__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       __half* __restrict__ wh, __half* __restrict__ wtc, float* __restrict__ wt, int64_t n, float lr,
                       float b1t, float b2t, const float* __restrict__ lparts, int n_l, float* __restrict__ loss)
{
    sum_loss(lparts, n_l, loss);
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / (1.f - b1t), vh = vi / (1.f - b2t);
    const float wi = w[i] - lr * mh / (sqrtf(vh) + eps);
    w[i] = wi;
    store_weight_copies(i, wi, wh, wtc, wt);
}

// every copy of the weights; zero: also the padding of the tensor-core tiles
// (features 524 to 575, which no weight fills)
__global__ void k_pack(const float* __restrict__ w, __half* __restrict__ wh, __half* __restrict__ wtc,
                       float* __restrict__ wt, int zero)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < kParams) store_weight_copies(i, w[i], wh, wtc, wt);
    if (zero && i < (int64_t)(kTcK1 - kIn) * kH) {
        const int n = (int)(i % kH), k = kIn + (int)(i / kH);
        wtc[(k / kTcChunk) * kTcW1Chunk + tc_off(n, k % kTcChunk, kTcChunk) / 2] = __float2half_rn(0.f);
    }
}

// predicted outer volume = fraction x cells
__global__ void k_pred_obv(const float* __restrict__ frac, const obb_qbox* __restrict__ boxes,
                           const int32_t* __restrict__ d_K, float* __restrict__ pred)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= *d_K) return;
    pred[i] = frac[i] * box_cells(boxes[i]);
}

// training target = exact outer volume / the same cell volume the screen scales by, in [0, 1]
__global__ void k_targets(const uint64_t* __restrict__ counts, const obb_qbox* __restrict__ boxes, int64_t K,
                          float* __restrict__ out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= K) return;
    const float cells = box_cells(boxes[i]);
    const float t = cells > 0.f ? (float)counts[i] / cells : 0.f;
    out[i] = fminf(fmaxf(t, 0.f), 1.f);
}

}  // namespace

struct MlpImpl {
    float* w = nullptr;    // FP32 master weights
    __half* wh = nullptr;  // FP16 inference copy
    __half* wtc = nullptr; // the FP16 weights transposed into the tensor-core kernel's shared tiles
    float* wt = nullptr;   // W2 and W3 transposed (the backward pass)
    float* g = nullptr;    // gradients
    float* m = nullptr;    // Adam moments
    float* v = nullptr;
    int64_t step = 0;
    int64_t cap = 0;       // batch capacity of the activation buffers
    float *h1 = nullptr, *h2 = nullptr, *h3 = nullptr, *y = nullptr, *d1 = nullptr, *d2 = nullptr, *d3 = nullptr,
          *dy = nullptr, *loss = nullptr, *lparts = nullptr;
};

}  // namespace obbv

struct obb_mlp {
    obb_ctx* ctx = nullptr;
    obbv::MlpImpl* p = nullptr;
};

namespace obbv {

// the context a network was created in (the entry points of other units
// check ownership through this; the type is complete only here)
const obb_ctx* mlp_owner(const obb_mlp* m) { return m ? m->ctx : nullptr; }

static obb_status mlp_reserve(obb_ctx* ctx, MlpImpl* P, int64_t B)
{
    if (B <= P->cap) return OBB_OK;
    cudaStream_t s = ctx->stream;
    float** bufs[] = {&P->h1, &P->h2, &P->h3, &P->d1, &P->d2, &P->d3};
    for (float** b : bufs) {
        if (*b) cudaFreeAsync(*b, s);
        OBB_CK(ctx, pool_alloc((void**)b, sizeof(float) * kH * B, s));
    }
    if (P->y) cudaFreeAsync(P->y, s);
    if (P->dy) cudaFreeAsync(P->dy, s);
    if (P->lparts) cudaFreeAsync(P->lparts, s);
    OBB_CK(ctx, pool_alloc((void**)&P->y, sizeof(float) * B, s));
    OBB_CK(ctx, pool_alloc((void**)&P->dy, sizeof(float) * B, s));
    OBB_CK(ctx, pool_alloc((void**)&P->lparts, sizeof(float) * ((B + 7) / 8), s));
    P->cap = B;
    return OBB_OK;
}

// rows a block of k_mlp_rows carries: 8 up to two blocks' worth an SM, else 16
static int rows_per_block(const obb_ctx* ctx, int B) { return B <= 16 * ctx->num_sms ? 8 : 16; }

template <int R, bool kTrain>
static cudaError_t launch_rows(obb_ctx* ctx, const MlpImpl* P, const float* X, int B, const int32_t* d_B,
                               const float* T, float* y, const RowsOut& out)
{
    const cudaError_t e = cudaFuncSetAttribute(k_mlp_rows<R, kTrain>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               rows_smem(R, kTrain));
    if (e != cudaSuccess) return e;
    k_mlp_rows<R, kTrain><<<(unsigned)((B + R - 1) / R), kRowsThreads, rows_smem(R, kTrain), ctx->stream>>>(
        X, B, d_B, P->w, P->wt, T, y, out);
    note_launch(ctx);
    return cudaGetLastError();
}

// forward pass into y (fraction); FP32 or FP16 weights
static obb_status mlp_forward(obb_ctx* ctx, const MlpImpl* P, const float* X, int B, const int32_t* d_B, bool half,
                              float* y)
{
    if (half) {
        // all four layers in one tensor-core kernel (FP16 operands, FP32 accumulators)
        cudaFuncSetAttribute(k_mlp_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, kTcSmem);
        const int32_t stall = (ctx->inject & OBB_INJECT_TC_STALL) ? 1 : 0;
        ctx->inject &= ~OBB_INJECT_TC_STALL;   // one launch only
        k_mlp_tc<<<(unsigned)((B + kTcRows - 1) / kTcRows), kTcRows, kTcSmem, ctx->stream>>>(X, B, d_B, P->wtc, P->wh,
                                                                                           P->w, y, ctx->d_err, stall);
        note_launch(ctx);
        OBB_CK(ctx, cudaGetLastError());
    } else if (rows_per_block(ctx, B) == 8) {
        OBB_CK(ctx, (launch_rows<8, false>(ctx, P, X, B, d_B, nullptr, y, RowsOut{})));
    } else {
        OBB_CK(ctx, (launch_rows<16, false>(ctx, P, X, B, d_B, nullptr, y, RowsOut{})));
    }
    return OBB_OK;
}

// gradients of the batch (FP32 weights) into P->g, the loss as *nl parts in P->lparts
static obb_status mlp_backward(obb_ctx* ctx, MlpImpl* P, const float* X, const float* T, int B, int* nl)
{
    const RowsOut out{P->h1, P->h2, P->h3, P->d1, P->d2, P->d3, P->dy, P->lparts};
    const int R = rows_per_block(ctx, B);
    if (R == 8) OBB_CK(ctx, (launch_rows<8, true>(ctx, P, X, B, nullptr, T, P->y, out)));
    else OBB_CK(ctx, (launch_rows<16, true>(ctx, P, X, B, nullptr, T, P->y, out)));
    *nl = (B + R - 1) / R;
    OBB_CK(ctx, cudaFuncSetAttribute(k_mlp_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, kGradSmem));
    k_mlp_wgrad<<<kGradBlocks, kGradThreads, kGradSmem, ctx->stream>>>(X, B, out, P->g);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

static void pack_weights(obb_ctx* ctx, MlpImpl* P, bool zero)
{
    k_pack<<<(unsigned)((kParams + 255) / 256), 256, 0, ctx->stream>>>(P->w, P->wh, P->wtc, P->wt, zero ? 1 : 0);
    note_launch(ctx);
}

obb_status surrogate_predict(obb_ctx* ctx, const obb_mlp* mlp, const obb_lattice* lat, const obb_qbox* d_boxes,
                             const int32_t* d_K, int64_t cap, float* d_feats, float* d_pred)
{
    MlpImpl* P = mlp->p;
    OBB_TRY(mlp_reserve(ctx, P, cap));
    launch_features(ctx, lat, d_boxes, d_K, cap, d_feats);
    OBB_TRY(mlp_forward(ctx, P, d_feats, (int)cap, d_K, true, P->y));
    k_pred_obv<<<(unsigned)((cap + 255) / 256), 256, 0, ctx->stream>>>(P->y, d_boxes, d_K, d_pred);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    return OBB_OK;
}

}  // namespace obbv

using namespace obbv;

namespace {
template <class T>
obb_status dev_in(obb_ctx* ctx, const T* src, size_t n, int on_device, void** hold, const T** out)
{
    if (on_device) {
        *out = src;
        return OBB_OK;
    }
    OBB_CK(ctx, pool_alloc(hold, sizeof(T) * n, ctx->stream));
    OBB_CK(ctx, cudaMemcpyAsync(*hold, src, sizeof(T) * n, cudaMemcpyHostToDevice, ctx->stream));
    *out = static_cast<const T*>(*hold);
    return OBB_OK;
}
}  // namespace

extern "C" {

obb_status obb_mlp_create(obb_ctx* ctx, uint64_t seed, obb_mlp** out)
{
    if (!ctx || !out) return fail(ctx, OBB_ERR_ARG, "null argument");
    *out = nullptr;
    // He-uniform initial weights from a seeded host generator, zero biases
    std::vector<float> w(kParams, 0.f);
    std::mt19937_64 rng(seed);
    auto fill = [&](int64_t off, int fan_in, int64_t count) {
        std::uniform_real_distribution<float> U(-std::sqrt(6.f / fan_in), std::sqrt(6.f / fan_in));
        for (int64_t i = 0; i < count; ++i) w[off + i] = U(rng);
    };
    fill(oW1, kIn, (int64_t)kIn * kH);
    fill(oW2, kH, (int64_t)kH * kH);
    fill(oW3, kH, (int64_t)kH * kH);
    fill(oW4, kH, kH);
    obb_mlp* m = new obb_mlp();
    m->ctx = ctx;
    m->p = new MlpImpl();
    MlpImpl* P = m->p;
    cudaStream_t s = ctx->stream;
    cudaError_t e = pool_alloc((void**)&P->w, sizeof(float) * kParams, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->wh, sizeof(__half) * kParams, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->wtc, sizeof(__half) * kTcPacked, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->wt, sizeof(float) * 2 * kH * kH, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->g, sizeof(float) * kParams, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->m, sizeof(float) * kParams, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->v, sizeof(float) * kParams, s);
    if (e == cudaSuccess) e = pool_alloc((void**)&P->loss, sizeof(float), s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(P->w, w.data(), sizeof(float) * kParams, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(P->m, 0, sizeof(float) * kParams, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(P->v, 0, sizeof(float) * kParams, s);
    if (e == cudaSuccess) {
        pack_weights(ctx, P, true);
        e = cudaStreamSynchronize(s);
    }
    if (e != cudaSuccess) {
        obb_mlp_free(m);
        return cuda_fail(ctx, e, "surrogate allocation");
    }
    *out = m;
    return OBB_OK;
}

void obb_mlp_free(obb_mlp* m)
{
    if (!m) return;
    cudaStream_t s = m->ctx ? m->ctx->stream : nullptr;
    if (m->p) {
        MlpImpl* P = m->p;
        void* ptrs[] = {P->w, P->wh, P->wtc, P->g, P->m, P->v, P->h1, P->h2, P->h3, P->y, P->d1, P->d2, P->d3, P->dy, P->loss, P->wt, P->lparts};
        for (void* q : ptrs)
            if (q) cudaFreeAsync(q, s);
        delete P;
    }
    delete m;
}

int64_t obb_mlp_num_params(void) { return kParams; }

obb_status obb_mlp_params(obb_ctx* ctx, const obb_mlp* m, float* out, int32_t on_device)
{
    if (!ctx || !m || !out) return fail(ctx, OBB_ERR_ARG, "null argument");
    if (m->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "network belongs to another context");
    OBB_CK(ctx, cudaMemcpyAsync(out, m->p->w, sizeof(float) * kParams,
                                on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, ctx->stream));
    return on_device ? OBB_OK : check_device_error(ctx);
}

obb_status obb_mlp_set_params(obb_ctx* ctx, obb_mlp* m, const float* in, int32_t on_device)
{
    if (!ctx || !m || !in) return fail(ctx, OBB_ERR_ARG, "null argument");
    if (m->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "network belongs to another context");
    MlpImpl* P = m->p;
    OBB_CK(ctx, cudaMemcpyAsync(P->w, in, sizeof(float) * kParams,
                                on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, ctx->stream));
    pack_weights(ctx, P, false);
    OBB_CK(ctx, cudaMemsetAsync(P->m, 0, sizeof(float) * kParams, ctx->stream));
    OBB_CK(ctx, cudaMemsetAsync(P->v, 0, sizeof(float) * kParams, ctx->stream));
    P->step = 0;
    return check_device_error(ctx);
}

obb_status obb_surrogate_features(obb_ctx* ctx, const obb_lattice* lat, const obb_qbox* boxes, int64_t K, float* feats,
                                  int32_t on_device)
{
    if (!ctx || !lat || (K > 0 && (!boxes || !feats))) return fail(ctx, OBB_ERR_ARG, "null argument");
    if (lat->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "lattice belongs to another context");
    if (K <= 0) return OBB_OK;
    void* hb = nullptr;
    const obb_qbox* db;
    OBB_TRY(dev_in(ctx, boxes, (size_t)K, on_device, &hb, &db));
    float* df = feats;
    if (!on_device) OBB_CK(ctx, pool_alloc((void**)&df, sizeof(float) * kIn * K, ctx->stream));
    launch_features(ctx, lat, db, nullptr, K, df);
    OBB_CK(ctx, cudaGetLastError());
    if (!on_device) {
        OBB_CK(ctx, cudaMemcpyAsync(feats, df, sizeof(float) * kIn * K, cudaMemcpyDeviceToHost, ctx->stream));
        cudaFreeAsync(df, ctx->stream);
    }
    if (hb) cudaFreeAsync(hb, ctx->stream);
    return on_device ? OBB_OK : check_device_error(ctx);
}

obb_status obb_surrogate_targets(obb_ctx* ctx, const obb_qbox* boxes, const uint64_t* counts, int64_t K, float* out,
                                 int32_t on_device)
{
    if (!ctx || (K > 0 && (!boxes || !counts || !out))) return fail(ctx, OBB_ERR_ARG, "null argument");
    if (K <= 0) return OBB_OK;
    void *hb = nullptr, *hc = nullptr;
    const obb_qbox* db;
    const uint64_t* dc;
    OBB_TRY(dev_in(ctx, boxes, (size_t)K, on_device, &hb, &db));
    OBB_TRY(dev_in(ctx, counts, (size_t)K, on_device, &hc, &dc));
    float* dout = out;
    if (!on_device) OBB_CK(ctx, pool_alloc((void**)&dout, sizeof(float) * K, ctx->stream));
    k_targets<<<(unsigned)((K + 255) / 256), 256, 0, ctx->stream>>>(dc, db, K, dout);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    if (!on_device) {
        OBB_CK(ctx, cudaMemcpyAsync(out, dout, sizeof(float) * K, cudaMemcpyDeviceToHost, ctx->stream));
        cudaFreeAsync(dout, ctx->stream);
    }
    if (hb) cudaFreeAsync(hb, ctx->stream);
    if (hc) cudaFreeAsync(hc, ctx->stream);
    return on_device ? OBB_OK : check_device_error(ctx);
}

obb_status obb_mlp_forward(obb_ctx* ctx, const obb_mlp* m, const float* feats, int64_t B, float* out,
                           int32_t half_weights, int32_t on_device)
{
    if (!ctx || !m || (B > 0 && (!feats || !out))) return fail(ctx, OBB_ERR_ARG, "null argument");
    if (m->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "network belongs to another context");
    if (B <= 0) return OBB_OK;
    if (B > (1 << 24)) return fail(ctx, OBB_ERR_RANGE, "batch too large");
    void* hx = nullptr;
    const float* dx;
    OBB_TRY(dev_in(ctx, feats, (size_t)B * kIn, on_device, &hx, &dx));
    OBB_TRY(mlp_reserve(ctx, m->p, B));
    float* y = on_device ? out : m->p->y;
    OBB_TRY(mlp_forward(ctx, m->p, dx, (int)B, nullptr, half_weights != 0, y));
    if (!on_device) OBB_CK(ctx, cudaMemcpyAsync(out, y, sizeof(float) * B, cudaMemcpyDeviceToHost, ctx->stream));
    if (hx) cudaFreeAsync(hx, ctx->stream);
    return on_device ? OBB_OK : check_device_error(ctx);
}

obb_status obb_mlp_gradients(obb_ctx* ctx, obb_mlp* m, const float* feats, const float* target, int64_t B,
                             float* grads, float* loss, int32_t on_device)
{
    if (!ctx || !m || !feats || !target || B <= 0) return fail(ctx, OBB_ERR_ARG, "bad argument");
    if (m->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "network belongs to another context");
    if (B > (1 << 24)) return fail(ctx, OBB_ERR_RANGE, "batch too large");
    void *hx = nullptr, *ht = nullptr;
    const float *dx, *dt;
    OBB_TRY(dev_in(ctx, feats, (size_t)B * kIn, on_device, &hx, &dx));
    OBB_TRY(dev_in(ctx, target, (size_t)B, on_device, &ht, &dt));
    OBB_TRY(mlp_reserve(ctx, m->p, B));
    MlpImpl* P = m->p;
    int nl;
    OBB_TRY(mlp_backward(ctx, P, dx, dt, (int)B, &nl));
    k_loss<<<1, 32, 0, ctx->stream>>>(P->lparts, nl, P->loss);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    if (grads) OBB_CK(ctx, cudaMemcpyAsync(grads, m->p->g, sizeof(float) * kParams, kind, ctx->stream));
    if (loss) OBB_CK(ctx, cudaMemcpyAsync(loss, m->p->loss, sizeof(float), kind, ctx->stream));
    if (hx) cudaFreeAsync(hx, ctx->stream);
    if (ht) cudaFreeAsync(ht, ctx->stream);
    return on_device ? OBB_OK : check_device_error(ctx);
}

obb_status obb_mlp_train_step(obb_ctx* ctx, obb_mlp* m, const float* feats, const float* target, int64_t B, float lr,
                              float* loss, int32_t on_device)
{
    if (!ctx || !m || !feats || !target || B <= 0) return fail(ctx, OBB_ERR_ARG, "bad argument");
    if (m->ctx != ctx) return fail(ctx, OBB_ERR_STATE, "network belongs to another context");
    if (B > (1 << 24)) return fail(ctx, OBB_ERR_RANGE, "batch too large");
    void *hx = nullptr, *ht = nullptr;
    const float *dx, *dt;
    OBB_TRY(dev_in(ctx, feats, (size_t)B * kIn, on_device, &hx, &dt));
    dx = dt;
    OBB_TRY(dev_in(ctx, target, (size_t)B, on_device, &ht, &dt));
    MlpImpl* P = m->p;
    OBB_TRY(mlp_reserve(ctx, P, B));
    int nl;
    OBB_TRY(mlp_backward(ctx, P, dx, dt, (int)B, &nl));
    P->step += 1;
    const float b1t = std::pow(0.9f, (float)P->step), b2t = std::pow(0.999f, (float)P->step);
    k_adam<<<(unsigned)((kParams + 255) / 256), 256, 0, ctx->stream>>>(P->w, P->g, P->m, P->v, P->wh, P->wtc, P->wt,
                                                                      kParams, lr, b1t, b2t, P->lparts, nl, P->loss);
    note_launch(ctx);
    OBB_CK(ctx, cudaGetLastError());
    if (loss)
        OBB_CK(ctx, cudaMemcpyAsync(loss, P->loss, sizeof(float),
                                    on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, ctx->stream));
    if (hx) cudaFreeAsync(hx, ctx->stream);
    if (ht) cudaFreeAsync(ht, ctx->stream);
    return (loss && !on_device) ? check_device_error(ctx) : OBB_OK;
}

}  // extern "C"
