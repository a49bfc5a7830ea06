// Device code of the exact outer-volume count (Eq. 4), shared by the kernels
// that count boxes: the per-box preparation and the counting of one tile of
// rows.  See outer_volume.cu for the method.
#pragma once

#include "internal.h"

#ifndef OBB_COUNT_UNROLL
#define OBB_COUNT_UNROLL 1
#endif
// OBB_BIG_TK_ROWS: boxes with at least this many (j, k) rows use tiles twice as tall (0: off)
#ifndef OBB_BIG_TK_ROWS
#define OBB_BIG_TK_ROWS 16384
#endif
// OBB_RANK_MIN_BITS: a box whose rows may be at least this long (in lattice
// points) is counted through the rank table; shorter rows (at most 64 points,
// two words) are counted from their two end words
#ifndef OBB_RANK_MIN_BITS
#define OBB_RANK_MIN_BITS 128
#endif
// OBB_ROW_MARGIN: rows added on each side of a box's (j, k) bounding rectangle
#ifndef OBB_ROW_MARGIN
#define OBB_ROW_MARGIN 1
#endif

namespace obbv {
// rint(2^24 rn(rn(r h_b) / hmax)): an entry of a box's integer normals
__device__ __noinline__ inline int32_t normal_exact(double r, const LatticeFrame* __restrict__ f, int b)
{
    return (int32_t)rint(__dmul_rn(__ddiv_rn(__dmul_rn(r, f->h[b]), f->hmax), 16777216.0));
}

// The same in integers: an FP64 instruction holds its scheduler for 64 cycles
// however many lanes take part (measured: a dependent chain and four
// independent ones both issue one in 64), and the defining sequence has
// thirteen.  With |r| < 2, x = floor(2^61 |r|) and y = x ratio / 2^64 is
// |r| h / hmax in units of 2^-60 within 258 of them (2^-53 of the ratio, the
// truncations); the rounded sequence is within 2^-52 of its value, 512 units.
// Farther than 4,096 units from a half-integer multiple of 2^36 both round to
// the same integer; else (1 entry in 2^23), or out of range, the sequence decides.
__device__ __forceinline__ int32_t normal_entry(double r, const LatticeFrame* __restrict__ f, int b)
{
    const uint64_t v = (uint64_t)__double_as_longlong(r);
    const int sh = 1014 - ((int)(v >> 52) & 0x7ff);   // |r| 2^61 = m 2^-sh
    if (sh >= -9) {
        const uint64_t m = (v & ((1ull << 52) - 1)) | (1ull << 52);
        const uint64_t x = sh <= 0 ? m << -sh : sh < 64 ? m >> sh : 0;
        const uint64_t y = __umul64hi(x, f->ratio[b]) + (1ull << 35);
        if ((y & ((1ull << 36) - 1)) - 4096 < (1ull << 36) - 8192) {
            const int32_t n = (int32_t)(y >> 36);
            return (int64_t)v < 0 ? -n : n;
        }
    }
    return normal_exact(r, f, b);
}

// unroll factor of the row loop, margin rows of a box's rectangle
constexpr int kCountUnroll = OBB_COUNT_UNROLL;
constexpr int kRowMargin = OBB_ROW_MARGIN;

namespace {

// The index axis along which a box is counted with the fewest rows: the one
// whose perpendicular plane receives the box's smallest shadow.  The shadow of
// the parallelepiped with edges e_a (columns of n^-1 scaled by H_a - L_a) on
// the plane of axes (s, t) has area sum_{a<b} |e_a,s e_b,t - e_a,t e_b,s|
// (FP32 from exact cofactors; ties to the lower axis).
__device__ __forceinline__ int choose_axis(const obb_qbox& q)
{
    int64_t m[9];
    for (int i = 0; i < 9; ++i) m[i] = q.n[i];
    const int64_t C[9] = {m[4] * m[8] - m[5] * m[7], m[2] * m[7] - m[1] * m[8], m[1] * m[5] - m[2] * m[4],
                          m[5] * m[6] - m[3] * m[8], m[0] * m[8] - m[2] * m[6], m[2] * m[3] - m[0] * m[5],
                          m[3] * m[7] - m[4] * m[6], m[1] * m[6] - m[0] * m[7], m[0] * m[4] - m[1] * m[3]};
    const __int128 det = (__int128)m[0] * C[0] + (__int128)m[1] * C[3] + (__int128)m[2] * C[6];
    if (det == 0) return 0;
    const float id = 1.0f / i128_to_float(det);
    float E[9];   // E[3 r + a]: component r of edge a
    for (int a = 0; a < 3; ++a) {
        const float d = i64_to_float((q.b[2 * a + 1] >> kS) - (-((-q.b[2 * a]) >> kS)));
        for (int r = 0; r < 3; ++r) E[3 * r + a] = i64_to_float(C[3 * r + a]) * id * d;
    }
    int best = 0;
    float best_area = 0.0f;
    for (int ax = 0; ax < 3; ++ax) {
        const int u = (ax + 1) % 3, v = (ax + 2) % 3;
        float area = 0.0f;
        for (int a = 0; a < 3; ++a)
            for (int b = a + 1; b < 3; ++b) area += fabsf(E[3 * u + a] * E[3 * v + b] - E[3 * v + a] * E[3 * u + b]);
        if (ax == 0 || area < best_area) {
            best = ax;
            best_area = area;
        }
    }
    return best;
}

// floor(x / d) and its remainder in [0, d), for 0 < d <= 2^24 and |x| < 2^62,
// by the integer reciprocal M = floor((2^64 - 1) / d): the high half of y M
// is at most one below floor(y / d) (M d > 2^64 - d - 1, y < 2^63), so one
// correction makes it exact.  All integer: 64-bit int <-> float conversions
// issue on the FP64 pipe, a small fraction of the integer rate on this GPU.
__device__ __forceinline__ void floordiv_rcp(int64_t x, int32_t d, uint64_t M, int64_t& q, int32_t& r)
{
    const bool neg = x < 0;
    const uint64_t y = neg ? (uint64_t)(-x) + (uint64_t)(d - 1) : (uint64_t)x;   // x < 0: floor(x/d) = -floor(y/d)
    uint64_t qq = __umul64hi(y, M);
    uint64_t rr = y - qq * (uint64_t)d;
    if (rr >= (uint64_t)d) {
        rr -= (uint64_t)d;
        ++qq;
    }
    q = neg ? -(int64_t)qq : (int64_t)qq;
    r = neg ? d - 1 - (int32_t)rr : (int32_t)rr;
}

// How a launch's boxes are counted: rows per lane per tile, row axis mode,
// rank rows on or off.
struct CountOpts {
    int32_t tile_k, axis_mode, count_rank;
};

// floor((2^64 - 1) / d) for 0 < d < 2^31: the high half by a 32-bit division;
// of the low half n / d, n = (rh + 1) 2^32 - 1, an FP32 estimate less 2,048 is
// never above it and less than 4,096 below (four roundings of 2^-24 of 2^32); the
// rest, below 2^12 d, once more, and a correction.
__device__ __forceinline__ uint64_t reciprocal64(uint32_t d)
{
    const uint32_t qh = 0xffffffffu / d, rh = 0xffffffffu - qh * d;
    const float inv = 1.0f / (float)d;
    const float est = (float)(rh + 1u) * inv * 4294967296.0f - 2048.0f;
    const uint32_t q0 = est > 0.0f ? (uint32_t)est : 0u;
    uint64_t r = ((uint64_t)rh << 32 | 0xffffffffu) - (uint64_t)q0 * d;
    // r beyond 32 bits only if d >= 2^20: the bits shifted out are less than 1 of the quotient
    const float f = (r >> 32) ? (float)(uint32_t)(r >> 12) * 4096.0f : (float)(uint32_t)r;
    const float e1 = f * inv - 2.0f;
    const uint32_t q1 = e1 > 0.0f ? (uint32_t)e1 : 0u;
    r -= (uint64_t)q1 * d;
    uint32_t q2 = 0;
    for (int i = 0; i < 6 && r >= d; ++i, r -= d) ++q2;   // three times at most over all 0 < d < 2^25
    return (uint64_t)qh << 32 | (uint64_t)(q0 + q1 + q2);
}

// Prepares box *qin of lattice lats[li] into *out and returns its number of
// tiles.  warps > 0: that many warps share the box; its tiles are cut so that
// each of them gets one (at least kMinTileRows rows a lane), since a lane
// walks its rows one after another and the rest of the machine would wait.
//
// Four lanes a box; the whole warp calls (qin null: nothing to do).  Lane a < 3
// computes what belongs to slab a and to index axis a, lane 3 repeats lane 0's
// part; they exchange through shuffles and hold the same box-wide values.  A
// preparation is one long chain of dependent instructions, which the callers
// wait for.  A lane a box against four lanes: five boxes on 64^3 11.5 -> 10.2 us
// in the kernel, flooding of 10,000 triangles 2.38 -> 1.89 ms, the rounds of
// 8,192 pairs 659 -> 572 us, the boxes of 98,304 probes 30.6 -> 20.0 us.
constexpr int32_t kMinTileRows = 4;   // 1 to 8 measure alike

__device__ __noinline__ int64_t prep_box(const obb_qbox* __restrict__ qin, int32_t li, const LatRef* __restrict__ lats,
                                         int32_t n_lats, const CountOpts o, int32_t warps,
                                         BoxPrep* __restrict__ out, int32_t* err)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 3;
    const int a = lane < 3 ? lane : 0;
    const bool on = qin != nullptr;
    const auto geti = [&](int32_t x, int from) { return __shfl_sync(kAll, x, from, 4); };
    const auto getf = [&](float x, int from) { return __shfl_sync(kAll, x, from, 4); };
    const bool bad_lat = li < 0 || li >= n_lats;
    if (bad_lat) li = 0;
    const LatRef& lr = lats[li];
    // count along the chosen axis: the index axes are relabelled (axis, then
    // the other two in order), which permutes the columns of n; the slab
    // bounds are unchanged.  A lattice without its y- and z-row copies is
    // counted along x.
    int32_t axis = 0;
    if (on && o.axis_mode != 0 && !bad_lat && lr.words_y) axis = o.axis_mode > 0 ? o.axis_mode : choose_axis(*qin);
    const auto entry = [&](int row, int c) {   // new axis c is old axis (axis, the others in order)[c]
        return on ? qin->n[3 * row + (c == 0 ? axis : (c <= axis ? c - 1 : c))] : 0;
    };
    const int32_t N = lr.N;
    const int32_t n0 = entry(a, 0), n1 = entry(a, 1), n2 = entry(a, 2);
    const int64_t L = on ? -((-qin->b[2 * a]) >> kS) : 0, H = on ? qin->b[2 * a + 1] >> kS : 0;
    const int32_t dd = n0 >= 0 ? n0 : -n0;
    // slab kind: 0 = n_a0 == 0 (a band in (y, z)), 1 = quotient DDA in 32 bits,
    // 2 = quotient DDA in 64 bits (|n_a0| < 32: the slab is almost parallel to x)
    const int32_t kind = n0 == 0 ? 0 : (dd >= 32 ? 1 : 2);
    int32_t mode = geti(kind, 0) | geti(kind, 1) << 2 | geti(kind, 2) << 4;
    const int32_t inverted = L > H;
    const int32_t any_inverted = geti(inverted, 0) | geti(inverted, 1) | geti(inverted, 2);   // every lane shuffles
    bool empty = bad_lat || any_inverted != 0;
    int32_t error = bad_lat ? kErrArg : 0;
    int32_t i0 = 0, span = -1, j0 = 0, k0 = 0, nj = 0, nk = 0;
    float nu_j = 0.0f, nu_k = 0.0f, sat_lo = -1.0f, sat_hi = 1.0f, kc_s = 0.0f, kc_lo = -1e30f, kc_hi = 1e30f;
    {
        // Exact cofactors of the integer normals (|n| <= 2^24: every product is
        // below 2^48) and the exact determinant in 128 bits; the geometry below
        // is FP32 with explicit margins (FP64 and 64-bit int <-> float
        // conversions issue on the FP64 pipe, a small fraction of the FP32
        // rate on this GPU).  Row a of the adjugate (M^-1 = C / det) comes from
        // the two other columns.
        const int u = a == 2 ? 0 : a + 1, v = a == 0 ? 2 : a - 1;
        int64_t mu[3], mv[3], C[3];
        for (int i = 0; i < 3; ++i) {
            mu[i] = entry(i, u);
            mv[i] = entry(i, v);
        }
        for (int i = 0; i < 3; ++i) C[i] = mu[(i + 1) % 3] * mv[(i + 2) % 3] - mv[(i + 1) % 3] * mu[(i + 2) % 3];
        const __int128 part = (__int128)(int64_t)entry(0, a) * C[0];
        __int128 det = 0;
        for (int r = 0; r < 3; ++r) {
            const uint64_t plo = __shfl_sync(kAll, (unsigned long long)part, r, 4);
            const int64_t phi = (int64_t)__shfl_sync(kAll, (long long)(part >> 64), r, 4);
            det += ((__int128)phi << 64) | (__int128)(unsigned __int128)plo;
        }
        if (!empty && det == 0) {
            error |= kErrArg;
            empty = true;
        }
        // FP32 inverse (relative error below 10 * 2^-24 per entry) and the
        // slab bounds: centre (L + H) / 2, half width (H - L) / 2, and
        // max(|L|, |H|), which bounds both
        const float id = 1.0f / i128_to_float(det);
        float mi[3];
        for (int i = 0; i < 3; ++i) mi[i] = i64_to_float(C[i]) * id;
        float yc[3], yh[3], ym[3], yl[3], yu[3];
        {
            const float l = i64_to_float(L), h = i64_to_float(H);
            const float c2 = 0.5f * i64_to_float(L + H), w2 = 0.5f * i64_to_float(H - L);
            for (int b = 0; b < 3; ++b) {
                yl[b] = getf(l, b);
                yu[b] = getf(h, b);
                yc[b] = getf(c2, b);
                yh[b] = getf(w2, b);
                ym[b] = fmaxf(fabsf(yl[b]), fabsf(yu[b]));
            }
        }
        // the parallelepiped {L <= M p <= H} has centre M^-1 (L + H) / 2 and
        // half extent sum_a |M^-1_ra| (H_a - L_a) / 2 along index axis r (this
        // lane's); the FP32 error of the two together is below 2e-6 of
        // sum_a |M^-1_ra| max(|L_a|, |H_a|), and the bounds are widened by
        // twice that
        float mn[3], mx[3];
        {
            float cen = 0.0f, ext = 0.0f, mag = 0.0f;
            for (int b = 0; b < 3; ++b) {
                const float w = mi[b];
                cen = fmaf(w, yc[b], cen);
                ext = fmaf(fabsf(w), yh[b], ext);
                mag = fmaf(fabsf(w), ym[b], mag);
            }
            const float e = 4e-6f * mag + 1e-3f;
            const float lo = cen - ext - e, hi = cen + ext + e;
            for (int r = 0; r < 3; ++r) {
                mn[r] = getf(lo, r);
                mx[r] = getf(hi, r);
            }
        }
        float m0[3], m1[3], m2[3];   // M^-1
        for (int b = 0; b < 3; ++b) {
            m0[b] = getf(mi[b], 0);
            m1[b] = getf(mi[b], 1);
            m2[b] = getf(mi[b], 2);
        }
        if (!empty) {
            const float lim = (float)kBoxRange;
            for (int r = 0; r < 3; ++r)
                if (!(mn[r] > -lim && mx[r] < lim + (float)N)) empty = true;
            const float span_j = mx[1] - mn[1] + 5.0f, span_k = mx[2] - mn[2] + 5.0f;
            if (!empty && span_j * span_k > 2.0e9f) empty = true;
            if (empty) error |= kErrRange;
        }
        if (!empty) {
            // beyond the widening above, a margin of two columns along x
            // and kRowMargin rows along y and z
            i0 = (int32_t)floorf(mn[0]) - 2;
            span = (int32_t)ceilf(mx[0]) + 2 - i0;
            j0 = (int32_t)floorf(mn[1]) - kRowMargin;
            const int32_t j1 = (int32_t)ceilf(mx[1]) + kRowMargin;
            k0 = (int32_t)floorf(mn[2]) - kRowMargin;
            const int32_t k1 = (int32_t)ceilf(mx[2]) + kRowMargin;
            nj = j1 - j0 + 1;
            nk = k1 - k0 + 1;
            // shadow on the (j, k) plane: edge a of the parallelepiped runs
            // along column a of M^-1; its normal nu_a in (j, k) is
            // orthogonal to that edge's shadow, and the shadow's extent
            // along nu_a is the sum over the other two constraints b of
            // nu_a . (column b) times [L_b, H_b].  Widened by two rows plus
            // 4e-6 of the terms' magnitude (the FP32 error, including the
            // neglected term of column a, is below 2e-6 of it).
            const float e0 = a == 0 ? m0[0] : a == 1 ? m0[1] : m0[2];
            const float e1 = a == 0 ? m1[0] : a == 1 ? m1[1] : m1[2];
            const float e2 = a == 0 ? m2[0] : a == 1 ? m2[1] : m2[2];
            float nj_ = -e2, nk_ = e1;
            const float len2 = nj_ * nj_ + nk_ * nk_;
            const float emax = fmaxf(fabsf(e0), fmaxf(fabsf(e1), fabsf(e2)));
            if (len2 > 1e-12f * emax * emax) {   // else the edge is parallel to x: no axis
                // (only the direction matters: the band below is computed
                // with this very normal, whatever its length)
                const float il = rsqrtf(len2);
                nj_ *= il;
                nk_ *= il;
                float lo = 0.0f, hi = 0.0f, mg = 0.0f;
                for (int b = 0; b < 3; ++b) {
                    mg = fmaf(fabsf(nj_ * m1[b]) + fabsf(nk_ * m2[b]), ym[b], mg);
                    if (b == a) continue;
                    const float w = nj_ * m1[b] + nk_ * m2[b];
                    const float x0 = w * yl[b], x1 = w * yu[b];
                    lo += fminf(x0, x1);
                    hi += fmaxf(x0, x1);
                }
                const float sm = 2.0f + 4e-6f * mg;
                nu_j = nj_;
                nu_k = nk_;
                sat_lo = lo - sm;
                sat_hi = hi + sm;
                // solved for k relative to (j0, k0), where the band is not
                // steep in k (|dk/dj| <= 64, so |nu_k| >= 1/65), with one
                // row plus 1e-5 of the terms' magnitude (above FP32 rounding
                // here and in the kernel's evaluation)
                if (fabsf(nj_) <= 64.0f * fabsf(nk_)) {
                    const float ivk = 1.0f / nk_;
                    const float sl = -nj_ * ivk;
                    const float b0 = (nk_ > 0.0f ? sat_lo : sat_hi) * ivk;
                    const float b1 = (nk_ > 0.0f ? sat_hi : sat_lo) * ivk;
                    const float fj0 = (float)j0, fk0 = (float)k0;
                    const float c0 = b0 + sl * fj0 - fk0, c1 = b1 + sl * fj0 - fk0;
                    const float mm = 1.0f + 1e-5f * (fabsf(sl) * (fabsf(fj0) + (float)nj) + fabsf(b0) + fabsf(b1) +
                                                     fabsf(fk0));
                    kc_s = sl;
                    kc_lo = c0 - mm;
                    kc_hi = c1 + mm;
                }
            }
        }
    }
    // rows per lane per tile: long tiles amortise the exact initial division
    // over more rows (set per context; obb_tune_counting picks it by timing)
    int32_t tk = o.tile_k;
#if OBB_BIG_TK_ROWS
    // boxes with many rows take tiles twice as tall (fewer tile setups; the
    // row clipping trims their empty ends)
    if ((int64_t)nj * nk >= OBB_BIG_TK_ROWS && 2 * o.tile_k <= 128) tk = 2 * o.tile_k;
#endif
    if (warps > 0) {   // nj nk <= 2e9, warps a small multiple of the SMs
        const uint32_t share = 32u * (uint32_t)warps;
        tk = min(tk, max(kMinTileRows, (int32_t)(((uint32_t)nj * (uint32_t)nk + share - 1) / share)));
    }
    // row counting: a box's rows are at most ell points long, the smallest of
    // span + 1 and (H_a - L_a) / |n_a0| + 1 over the slabs that step along x.
    // With rank tables, long rows (ell >= OBB_RANK_MIN_BITS) are counted from
    // their two end words and the rank table, and rows of at most 64 points
    // (ell < 63.5, well clear of FP32 rounding) from their two end words; both
    // at a fixed cost per row.
    const uint16_t* const ranks = axis == 0 ? lr.rank : (axis == 1 ? lr.rank_y : lr.rank_z);
    int32_t rank = 0;
    {
        const float own = dd > 0 ? i64_to_float(H - L) / (float)dd + 1.0f : 3.0e38f;
        float ell = fminf((float)span + 1.0f, (float)N);
        for (int b = 0; b < 3; ++b) ell = fminf(ell, getf(own, b));
        if (nj > 0 && o.count_rank && ranks) rank = ell >= (float)OBB_RANK_MIN_BITS ? 1 : (ell < 63.5f ? 2 : 0);
    }
    // tile shape: wj lanes along y, wk = 32 / wj along z; the least padding wins
    // (ties to the wider wj, whose rows sit next to each other in memory); a
    // lane tries two of the six
    int best = 5;
    {
        // ceil(nk / ((32 >> l) tk)) = ceil(ceil(nk / tk) / 2^(5 - l)): one division
        const int32_t nkt = (nk + tk - 1) / tk;
        int64_t key = INT64_MAX;
        for (int sh = lane; sh < 6; sh += 4) {
            const int l = 5 - sh;
            const int64_t slots = (int64_t)(((nj + (1 << l) - 1) >> l) << l) *
                                  ((int64_t)((nkt + (1 << sh) - 1) >> sh) * ((32 >> l) * tk));
            key = min(key, slots << 3 | sh);
        }
        for (int x = 1; x < 4; x <<= 1) key = min(key, (int64_t)__shfl_xor_sync(kAll, (long long)key, x));
        if (nj > 0) best = 5 - (int)(key & 7);
    }
    // interior box: its whole index rectangle lies in the lattice, so no row
    // and no x-interval needs clamping to [0, N)
    if (nj > 0 && i0 >= 0 && i0 + span <= N - 1 && j0 >= 0 && j0 + nj <= N && k0 >= 0 && k0 + nk <= N) mode |= 1 << 8;
    const int32_t wj = 1 << best, wk = 32 >> best;
    const int32_t ntj = nj > 0 ? (nj + wj - 1) / wj : 0;
    int32_t qs = 0, rs = 0, rw = 0;
    uint64_t M = 0;
    int64_t fstep = 0, qw = 0;
    if (kind != 0) {
        // between a lane's rows k advances by wk: X_lo and X_hi move by -sign(d) * n_a2 * wk
        // |delta| <= 2^24 * 32 and 0 < dd < 2^25: exact in 32 bits
        const int32_t delta = -(n0 > 0 ? 1 : -1) * n2 * wk;
        qs = delta / dd;
        if (qs * dd > delta) --qs;   // floor
        rs = delta - qs * dd;
        // the same step in 32.32 fixed point, rounded down (exact division:
        // rstep < dd <= 2^24, so rstep * 2^32 < 2^56)
        M = reciprocal64((uint32_t)dd);
        // floor(rstep 2^32 / dd) through the reciprocal: rstep M / 2^32 is
        // less than 2^-8 below it, so its floor is exact or one short
        const uint32_t ru = (uint32_t)rs;
        uint64_t fr = (uint64_t)ru * (uint32_t)(M >> 32) + __umulhi(ru, (uint32_t)M);
        if ((fr + 1) * (uint64_t)dd <= ((uint64_t)ru << 32)) ++fr;
        fstep = (int64_t)qs * 4294967296LL + (int64_t)fr;
        floordiv_rcp(H - L - dd + 1, dd, M, qw, rw);
    }
    // A quotient saturated at +-2^30 must stay outside [0, span] for a whole
    // tile: its tk - 1 steps of at most |qstep| + 1 each stay below 2^29.  With
    // |qstep| <= 2^24 every tk <= 32 qualifies; taller tiles are cut for steep
    // slabs.
    {
        const int32_t own = kind == 1 ? abs(qs) + 1 : 0;
        const int32_t smax = max(geti(own, 0), max(geti(own, 1), geti(own, 2)));
        if (smax > 0 && (int64_t)(tk - 1) * smax >= (int64_t(1) << 29)) tk = max(1, min(tk, (1 << 29) / smax));
    }
    // A warp adds up its tile's points in 32 bits: 32 lanes, tk rows each, rows
    // of at most span + 1 points.  Only rows beyond 2^20 points cut a tile.
    if ((int64_t)tk * (span + 1) >= (int64_t(1) << 27)) tk = ((1 << 27) - 1) / (span + 1);
    if (!on) return 0;
    if (lane < 3) {
        out->sat_nu[a][0] = nu_j;
        out->sat_nu[a][1] = nu_k;
        out->sat_lo[a] = sat_lo;
        out->sat_hi[a] = sat_hi;
        out->kc_s[a] = kc_s;
        out->kc_lo[a] = kc_lo;
        out->kc_hi[a] = kc_hi;
        out->n[3 * a] = n0;
        out->n[3 * a + 1] = n1;
        out->n[3 * a + 2] = n2;
        out->dd[a] = dd;
        out->Lq[a] = L;
        out->Hq[a] = H;
        out->fmul[a] = M;
        out->qw[a] = qw;
        out->rw[a] = rw;
        out->fstep[a] = fstep;
        out->rstep[a] = rs;
        out->qstep[a] = qs;
    } else {
        if (error) atomicOr(err, error);
        out->words = axis == 0 ? lr.words : (axis == 1 ? lr.words_y : lr.words_z);
        out->ranks = ranks;
        out->latN = N;
        out->latW = lr.W;
        out->ntj = ntj;
        out->lwj = best;
        out->tk = tk;
        out->mode = mode;
        out->j0 = j0;
        out->k0 = k0;
        out->nj = nj;
        out->nk = nk;
        out->i0 = i0;
        out->span = span;
        out->axis = axis;
        out->lat = li;
        out->rank = rank;
    }
    return nj > 0 ? (int64_t)ntj * ((nk + wk * tk - 1) / (wk * tk)) : 0;
}

// 32.32 fixed-point DDA.  A slab bound floor(v), v = q + r / dd, is carried as
// A = q 2^32 + floor(r M / 2^32) + kFixBias with M = floor((2^64 - 1) / dd),
// and steps by floor(s 2^32) per row (s the exact rational step).  The seed is
// at most 1 + 2^-8 units (of 2^-32) below v 2^32 and never above it; each
// step loses less than one unit.  After r <= 127 steps the error lies in
// (kFixBias - 1 - 2^-8 - r, kFixBias] = (1.99, 130]: positive, and below
// 2^32 / dd >= 256, the distance from the largest fraction (dd - 1) / dd to
// the next integer.  So A >> 32 is exactly floor(v) on every row of a tile
// of at most 128 rows (the most obb_set_counting_tile allows).
constexpr int64_t kFixBias = 130;

__device__ __forceinline__ int64_t fixed_frac(int32_t r, uint64_t M)   // 0 <= r < 2^24
{
    const uint32_t ru = (uint32_t)r;
    return (int64_t)((uint64_t)ru * (uint32_t)(M >> 32) + __umulhi(ru, (uint32_t)M));
}

// Intersect [lo, hi] with { i : L <= d i + c <= H } exactly (d != 0), by
// integer-reciprocal division (M = floor((2^64 - 1) / |d|)).  Used per row for
// slabs almost parallel to x.
__device__ __forceinline__ void clip_slab_rcp(int32_t d, uint64_t M, int64_t c, int64_t L, int64_t H, int32_t& lo,
                                              int32_t& hi)
{
    const int32_t dd = d > 0 ? d : -d;
    const int64_t A = d > 0 ? L - c : c - H;
    const int64_t B = d > 0 ? H - c : c - L;
    int64_t qn, qb;
    int32_t rem;
    floordiv_rcp(-A, dd, M, qn, rem);   // ceil(A / dd) = -floor(-A / dd)
    floordiv_rcp(B, dd, M, qb, rem);
    const int64_t g = min(max(-qn, (int64_t)lo), (int64_t)hi + 1);
    const int64_t u = max(min(qb, (int64_t)hi), (int64_t)lo - 1);
    lo = (int32_t)g;
    hi = (int32_t)u;
}

// popcount of the occupied bits i in [a, e] of one row (0 <= a <= e < N) of
// a counting copy, the row's word w at row[w ws] (ws = N, the copy's column
// interleave); 64-bit words: the first and last word carry the masks (merged
// without a branch when they are the same word), interior words count whole.
__device__ __forceinline__ uint32_t popc_range(const uint64_t* __restrict__ row, int32_t ws, int32_t a, int32_t e)
{
    const int32_t wa = a >> 6, we = e >> 6;
    const uint64_t first = __ldg(row + wa * ws);
    const uint64_t last = __ldg(row + we * ws);
    uint64_t mlo = ~0ull << (a & 63);
    const uint64_t mhi = ~0ull >> (63 - (e & 63));
    uint32_t cnt = 0;
    for (int32_t w = wa + 1; w < we; ++w) cnt += __popcll(__ldg(row + w * ws));
    const bool one = wa == we;
    mlo = one ? (mlo & mhi) : mlo;
    return cnt + __popcll(first & mlo) + __popcll(last & (one ? 0ull : mhi));
}

// bits of the end words up to e, less those before a (mod 2^32)
__device__ __forceinline__ uint32_t rank_bits(uint64_t first, uint64_t last, int32_t a, int32_t e)
{
    return (uint32_t)__popcll(last << (~e & 63)) - (uint32_t)__popcll(first & ~(~0ull << (a & 63)));
}

// The same count through the row's rank table (rk[w ws] = occupied bits in
// words 0..w-1): the bits before e + 1 minus the bits before a, each a rank
// entry plus the popcount of its word below the bit -- four loads whatever
// the row's length, and no case for an interval inside one word.
__device__ __forceinline__ uint32_t popc_rank(const uint64_t* __restrict__ row, const uint16_t* __restrict__ rk,
                                              int32_t ws, int32_t a, int32_t e)
{
    const int32_t wa = a >> 6, we = e >> 6;
    const uint64_t first = __ldg(row + wa * ws);
    const uint64_t last = __ldg(row + we * ws);
    const uint32_t ra = __ldg(rk + wa * ws), rb = __ldg(rk + we * ws);
    return rb - ra + rank_bits(first, last, a, e);
}

// occupied bits of [a, e] from its two end words, when it has no others: the
// bits from a on and those up to e (shifts, no masks); in one word, less all
__device__ __forceinline__ uint32_t short_bits(uint64_t first, uint64_t last, int32_t a, int32_t e)
{
    return __popcll(first >> (a & 63)) + __popcll(last << (~e & 63)) - ((a ^ e) < 64 ? __popcll(first) : 0);
}

// occupied bits of [a, e] when it lies within two consecutive words
__device__ __forceinline__ uint32_t popc_short(const uint64_t* __restrict__ row, int32_t ws, int32_t a, int32_t e)
{
    const int32_t wa = a >> 6, we = e >> 6;
    const uint64_t first = __ldg(row + wa * ws);
    const uint64_t last = __ldg(row + we * ws);
    return short_bits(first, last, a, e);
}

// Row counting modes of a box (BoxPrep::rank).
enum { kRowWalk = 0, kRowRank = 1, kRowShort = 2 };

// algorithmic bytes of one counted row [a, e]: every 16-byte chunk the
// interval touches; through the rank table, the end words' chunks and two
// 2-byte rank entries
template <int kMode>
__device__ __forceinline__ uint32_t row_bytes(int32_t a, int32_t e)
{
    const int32_t ca = a >> 7, ce = e >> 7;
    return kMode == kRowRank ? (ca == ce ? 16u : 32u) + 4u : (uint32_t)(ce - ca + 1) * 16u;
}

// occupied bits of [a, e] by the box's row counting mode
template <int kMode>
__device__ __forceinline__ uint32_t popc_mode(const uint64_t* __restrict__ row, const uint16_t* __restrict__ rk,
                                              int32_t ws, int32_t a, int32_t e)
{
    if constexpr (kMode == kRowRank) return popc_rank(row, rk, ws, a, e);
    else if constexpr (kMode == kRowShort) return popc_short(row, ws, a, e);
    else return popc_range(row, ws, a, e);
}

// The first row's interval of a lane, relative to i0, from the six bounds of
// the DDA; the bounds step to the next row.
__device__ __forceinline__ void dda_step(int64_t (&Al)[3], int64_t (&Ah)[3], const int64_t (&Bs)[3], int32_t span,
                                         int32_t& lo, int32_t& hi)
{
    lo = max(max((int32_t)(Al[0] >> 32), (int32_t)(Al[1] >> 32)), max((int32_t)(Al[2] >> 32), 0));
    hi = min(min((int32_t)(Ah[0] >> 32), (int32_t)(Ah[1] >> 32)), min((int32_t)(Ah[2] >> 32), span));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Al[a] += Bs[a];
        Ah[a] += Bs[a];
    }
}

// One pass of a lane over its rows r0..r1 of a tile of a box whose three
// slabs all step by DDA: each of the six bounds is a 32.32 fixed-point value
// whose integer part is the quotient, so a bound costs one 64-bit add per
// row.  The loop is bound by issue slots, most of them integer ones: a row's
// place is a 32-bit offset (at, mod 2^32: rows outside the lattice are not
// read, and the largest copy has 2^27 words) and the bits are counted by
// shifts where a mask can be saved.  32,767 tree boxes at 1024^3: 257 us, 285
// with 64-bit row pointers, masks, two divisions a slab and the in-domain
// points of interior rows added up twice.
//
// dda_interior: rows whose words are the two at their ends (kMode kRowRank or
// kRowShort) of a tile that lies in the lattice with all of its x-intervals
// (an idle lane's span is -1).  A row's words are counted a row later, behind
// the next row's bounds (261 -> 257 us).
template <int kMode, bool kProf>
__device__ __forceinline__ void dda_interior(int64_t (&Al)[3], int64_t (&Ah)[3], const int64_t (&Bs)[3],
                                             const uint64_t* __restrict__ words, const uint16_t* __restrict__ ranks,
                                             uint32_t at, uint32_t rstride, int32_t rows, int32_t i0, int32_t span,
                                             int32_t N, uint32_t& empty, uint32_t& inbox, uint32_t& my_bytes,
                                             uint32_t& my_rows, uint32_t& my_rank, uint32_t& my_dom)
{
    uint32_t in = 0, occ = 0, rk = 0;
    uint64_t first = 0, last = 0;
    int32_t a = 0, e = 0;
    const auto take = [&] {
        occ += kMode == kRowRank ? rk + rank_bits(first, last, a, e) : short_bits(first, last, a, e);
    };
    for (int32_t r = 0; r < rows; ++r, at += rstride) {
        int32_t lo, hi;
        dda_step(Al, Ah, Bs, span, lo, hi);
        take();
        first = last = 0;
        rk = 0;
        if (lo <= hi) {
            a = i0 + lo;
            e = i0 + hi;
            in += (uint32_t)(hi - lo + 1);
            const uint32_t pa = at + (a >> 6) * N, pe = at + (e >> 6) * N;
            first = __ldg(words + pa);
            last = __ldg(words + pe);
            if (kMode == kRowRank) rk = (uint32_t)__ldg(ranks + pe) - (uint32_t)__ldg(ranks + pa);
            if (kProf) {
                my_bytes += row_bytes<kMode>(a, e);
                my_rows += 1;
                my_rank += kMode == kRowRank ? 1u : 0u;
            }
        }
    }
    take();
    inbox += in;
    empty += in - occ;
    my_dom += in;
}

// dda_rows: any other tile.  kInterior: as above, with words between the ends.
template <int kMode, bool kInterior, bool kProf>
__device__ __forceinline__ void dda_rows(int64_t (&Al)[3], int64_t (&Ah)[3], const int64_t (&Bs)[3],
                                         const uint64_t* __restrict__ words, const uint16_t* __restrict__ ranks,
                                         uint32_t at, uint32_t rstride, int32_t rows, int32_t k, int32_t wk,
                                         int32_t kend, bool jvalid, bool jin, int32_t i0, int32_t span, int32_t N,
                                         uint32_t& empty, uint32_t& inbox, uint32_t& my_bytes, uint32_t& my_rows,
                                         uint32_t& my_rank, uint32_t& my_dom)
{
#pragma unroll kCountUnroll
    for (int32_t r = 0; r < rows; ++r, k += wk, at += rstride) {
        int32_t lo, hi;
        dda_step(Al, Ah, Bs, span, lo, hi);
        if (kInterior ? lo <= hi : jvalid && k < kend && lo <= hi) {
            const uint32_t len = (uint32_t)(hi - lo + 1);
            uint32_t occ = 0;
            if (kInterior || (jin && (uint32_t)k < (uint32_t)N)) {
                const int32_t a = kInterior ? i0 + lo : max(i0 + lo, 0), e = kInterior ? i0 + hi : min(i0 + hi, N - 1);
                if (kInterior || a <= e) {
                    occ = popc_mode<kMode>(words + at, ranks + at, N, a, e);
                    my_dom += (uint32_t)(e - a + 1);
                    if (kProf) my_bytes += row_bytes<kMode>(a, e);
                }
            }
            empty += len - occ;
            inbox += len;
            if (kProf) {
                my_rows += 1;
                my_rank += kMode == kRowRank ? 1u : 0u;
            }
        }
    }
}

// Counts tile (tj, tk) of box p: the calling warp adds its lanes' empty and
// all points of the box to empty and inbox (not yet summed over the warp), and
// its in-domain points to my_dom (kProf: also the algorithmic bytes, rows and
// rank rows).  False: the box's shadow misses the tile.
template <bool kProf>
__device__ __forceinline__ bool count_tile(const BoxPrep& p, int32_t tj, int32_t tk, uint32_t& empty, uint32_t& inbox,
                                           uint32_t& my_bytes, uint32_t& my_rows, uint32_t& my_rank, uint32_t& my_dom)
{
    const int lane = threadIdx.x & 31;
    {
        // skip a tile whose rectangle misses the box's shadow on (j, k)
        const int32_t lw = p.lwj, hk = (32 >> lw) * p.tk;
        const float hj = 0.5f * (float)((1 << lw) - 1), hkf = 0.5f * (float)(hk - 1);
        const float jc = (float)(p.j0 + (tj << lw)) + hj, kc = (float)(p.k0 + tk * hk) + hkf;
        bool out = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float u = p.sat_nu[a][0], v = p.sat_nu[a][1];
            const float cc = u * jc + v * kc, e = fabsf(u) * hj + fabsf(v) * hkf;
            out |= cc + e < p.sat_lo[a] || cc - e > p.sat_hi[a];
        }
        if (out) return false;
    }
    const uint64_t* __restrict__ words = p.words;
    const int32_t N = p.latN, W = p.latW;
    const int32_t mode = p.mode;
    const int32_t lwj = p.lwj;
    const int32_t wk = 32 >> lwj;
    const int32_t jl = (tj << lwj) + (lane & ((1 << lwj) - 1));
    const int32_t j = p.j0 + jl;
    const bool jvalid = jl < p.nj;
    const int32_t tkr = p.tk;
    const int32_t kb = p.k0 + tk * (wk * tkr) + (lane >> lwj);   // this lane's first row
    const int32_t kend = p.k0 + p.nk;
    // rows r0..r1 (warp-uniform) of the tile's tkr are visited
    int32_t r0 = 0, r1 = tkr - 1;
    if ((mode & 0xff) == 0x15) {
        // each lane's column meets the shadow in a k-range (the separating
        // bands solved for k); the warp visits the union of its lanes'
        // ranges, which skips the empty ends of a tile the shadow crosses
        const float jr = (float)(j - p.j0);
        float klo = -1e30f, khi = 1e30f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            klo = fmaxf(klo, fmaf(p.kc_s[a], jr, p.kc_lo[a]));
            khi = fminf(khi, fmaf(p.kc_s[a], jr, p.kc_hi[a]));
        }
        int32_t rl = tkr, rh = -1;
        if (jvalid && klo <= khi) {
            const int32_t lwk = 5 - lwj;   // wk = 2^lwk
            const int32_t kbr = kb - p.k0;
            const int32_t kl = (int32_t)floorf(fmaxf(klo, -1e9f));
            const int32_t kh = (int32_t)ceilf(fminf(khi, 1e9f));
            rl = max(0, -((kbr - kl) >> lwk));    // first r with kb + r wk >= kl
            rh = min(tkr - 1, (kh - kbr) >> lwk);  // last r with kb + r wk <= kh
            if (rl > rh) {
                rl = tkr;
                rh = -1;
            }
        }
        r0 = __reduce_min_sync(0xffffffffu, rl);
        r1 = __reduce_max_sync(0xffffffffu, rh);
        if (r0 > r1) return false;
    }
    const int32_t kb0 = kb + r0 * wk;   // the first row this lane visits
    const int32_t i0 = p.i0, span = p.span;
    // Kind-1 slabs carry exact quotient bounds relative to i0 in 32 bits,
    // saturated at +-2^30: a bound that far out moves less than 2^29 within a
    // tile, so it stays outside [0, span].  Kind 0 (n_a0 = 0) and kind 2
    // (|n_a0| < 32) slabs are evaluated from scratch on each row.
    int32_t qa[3], qb[3], ra[3], rb[3], dd[3], rs[3], qs[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        qa[a] = qb[a] = ra[a] = rb[a] = rs[a] = qs[a] = 0;
        dd[a] = 1;
        if (((mode >> (2 * a)) & 3) == 1) {
            dd[a] = p.dd[a];
            rs[a] = p.rstep[a];
            qs[a] = p.qstep[a];
            const int64_t cc = (int64_t)p.n[3 * a + 1] * j + (int64_t)p.n[3 * a + 2] * kb0;
            const int64_t xlo = p.n[3 * a] > 0 ? p.Lq[a] - cc : cc - p.Hq[a];
            int64_t wlo;
            floordiv_rcp(xlo + dd[a] - 1, dd[a], p.fmul[a], wlo, ra[a]);   // ceil(xlo / dd)
            // the upper bound floor(xhi / dd): xhi = (xlo + dd - 1) + (H - L - dd + 1)
            int64_t whi = wlo + p.qw[a];
            rb[a] = ra[a] + p.rw[a];
            if (rb[a] >= dd[a]) {
                rb[a] -= dd[a];
                ++whi;
            }
            const int64_t lim = int64_t(1) << 30;
            qa[a] = (int32_t)min(max(wlo - i0, -lim), lim);
            qb[a] = (int32_t)min(max(whi - i0, -lim), lim);
        }
    }
    const bool jin = j >= 0 && j < N;
    if ((mode & 0xff) == 0x15) {
        // all three slabs step by DDA (any rotated box): the 32.32
        // fixed-point bounds, seeded exactly at the first visited row
        int64_t Al[3], Ah[3], Bs[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const uint64_t M = p.fmul[a];
            Al[a] = (int64_t)qa[a] * 4294967296LL + fixed_frac(ra[a], M) + kFixBias;
            Ah[a] = (int64_t)qb[a] * 4294967296LL + fixed_frac(rb[a], M) + kFixBias;
            Bs[a] = p.fstep[a];
        }
        // count copies interleave the rows of a slice by column: word w of
        // row (slice k, column j) at (k W + w) N + j
        const uint32_t at = (uint32_t)kb0 * (uint32_t)(W * N) + (uint32_t)j;
        const uint32_t rstride = (uint32_t)wk * (uint32_t)(W * N);
        const int32_t rows = r1 - r0 + 1;
        // an interior box's full-height tile: every row is in the lattice
        // and so is every x-interval; an idle lane gets an empty range
        const bool interior = (mode & 0x100) && (tk + 1) * wk * tkr <= p.nk;
        const int32_t spanl = jvalid ? span : -1;
#define OBB_DDA_INTERIOR(MODE)                                                                                       \
dda_interior<MODE, kProf>(Al, Ah, Bs, words, p.ranks, at, rstride, rows, i0, spanl, N, empty, inbox, my_bytes, my_rows, \
                          my_rank, my_dom)
#define OBB_DDA_ROWS(MODE, INTERIOR)                                                                               \
dda_rows<MODE, INTERIOR, kProf>(Al, Ah, Bs, words, p.ranks, at, rstride, rows, kb0, wk, kend, jvalid, jin, i0,       \
                                INTERIOR ? spanl : span, N, empty, inbox, my_bytes, my_rows, my_rank, my_dom)
        if (p.rank == kRowRank) {
            if (interior) OBB_DDA_INTERIOR(kRowRank);
            else OBB_DDA_ROWS(kRowRank, false);
        } else if (p.rank == kRowShort) {
            if (interior) OBB_DDA_INTERIOR(kRowShort);
            else OBB_DDA_ROWS(kRowShort, false);
        } else {
            if (interior) OBB_DDA_ROWS(kRowWalk, true);
            else OBB_DDA_ROWS(kRowWalk, false);
        }
#undef OBB_DDA_INTERIOR
#undef OBB_DDA_ROWS
    } else
#pragma unroll kCountUnroll
    for (int r = 0; r < tkr; ++r) {
        const int32_t k = kb + r * wk;
        int32_t lo = 0, hi = span;
        bool ok = jvalid && k < kend;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int kind = (mode >> (2 * a)) & 3;
            if (kind == 1) {
                lo = max(lo, qa[a]);
                hi = min(hi, qb[a]);
                qa[a] += qs[a];
                ra[a] += rs[a];
                if (ra[a] >= dd[a]) {
                    ra[a] -= dd[a];
                    qa[a] += 1;
                }
                qb[a] += qs[a];
                rb[a] += rs[a];
                if (rb[a] >= dd[a]) {
                    rb[a] -= dd[a];
                    qb[a] += 1;
                }
            } else if (ok && lo <= hi) {
                const int64_t cc = (int64_t)p.n[3 * a + 1] * j + (int64_t)p.n[3 * a + 2] * k;
                if (kind == 0) {
                    ok = cc >= p.Lq[a] && cc <= p.Hq[a];
                } else {
                    int32_t l2 = i0 + lo, h2 = i0 + hi;
                    clip_slab_rcp(p.n[3 * a], p.fmul[a], cc, p.Lq[a], p.Hq[a], l2, h2);
                    lo = l2 - i0;
                    hi = h2 - i0;
                }
            }
        }
        if (ok && lo <= hi) {
            const int32_t ia = i0 + lo, ie = i0 + hi;
            const uint32_t len = (uint32_t)(hi - lo + 1);
            uint32_t occ = 0;
            if (jin && k >= 0 && k < N) {
                const int32_t a = max(ia, 0), e = min(ie, N - 1);
                if (a <= e) {
                    const int64_t roff = (int64_t)k * W * N + j;
                    if (p.rank == kRowRank) {
                        occ = popc_rank(words + roff, p.ranks + roff, N, a, e);
                        if (kProf) my_bytes += row_bytes<kRowRank>(a, e);
                    } else {
                        occ = popc_range(words + roff, N, a, e);
                        if (kProf) my_bytes += row_bytes<kRowWalk>(a, e);
                    }
                    my_dom += (uint32_t)(e - a + 1);
                }
            }
            empty += len - occ;
            inbox += len;
            if (kProf) {
                my_rows += 1;
                my_rank += p.rank == kRowRank ? 1u : 0u;
            }
        }
    }
    return true;
}

}  // namespace
}  // namespace obbv
