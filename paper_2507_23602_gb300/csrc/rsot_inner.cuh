// Inner loops of the mixed-precision passes, shared by the single-problem,
// allocation-free and batched kernels.  Log2 domain: for a point x' and a
// target record (w_j, c_j), r_qj = c_j + x'.w_j (see rsot_dense.cu).
#pragma once

#include "rsot_internal.cuh"

namespace rsot {

// Tile shapes; the build may override them (-DRSOT_P1_PP=..., etc.) to tune.
#ifndef RSOT_P1_PP
#define RSOT_P1_PP 4
#endif
#ifndef RSOT_P1_MINB
#define RSOT_P1_MINB 4
#endif
#ifndef RSOT_P1_SUB
#define RSOT_P1_SUB 16
#endif
#ifndef RSOT_P2_MINB
#define RSOT_P2_MINB 1
#endif
#ifndef RSOT_P2_TPP
#define RSOT_P2_TPP 4
#endif
inline constexpr int P1_THREADS = 128;
inline constexpr int P1_PP = RSOT_P1_PP;                      // point pairs per thread (<= 4)
inline constexpr int P1_TILE = P1_THREADS * 2 * P1_PP;        // points per CTA (divides 1024)
inline constexpr int P1_MINB = RSOT_P1_MINB;                  // resident CTAs per SM asked of ptxas
__host__ __device__ constexpr int p1_minb(int pp) { return pp == 4 ? P1_MINB : pp == 2 ? 2 * P1_MINB : 12; }
#ifndef RSOT_P1_TS
#define RSOT_P1_TS 512
#endif
#ifndef RSOT_P2_TS
#define RSOT_P2_TS 512
#endif
inline constexpr int P1_TS = RSOT_P1_TS;                      // targets per stage (divides 1024)
inline constexpr int P1_STAGES = 2;
inline constexpr int P1_SUB = RSOT_P1_SUB;                    // targets per optimistic sub-tile
inline constexpr int P2_MINB = RSOT_P2_MINB;
inline constexpr int P2_TPP_MAX = RSOT_P2_TPP;                // target pairs per thread (pass 2)
inline constexpr float P1_BIG = 1.152921504606846976e18f;     // 2^60: a sub-tile sum above it is redone

inline constexpr int P2_THREADS = 128;
inline constexpr int P2_TS = RSOT_P2_TS;                      // points per stage (divides 1024)
static_assert(1024 % P1_TS == 0 && 1024 % P2_TS == 0 && P1_TS % P1_SUB == 0, "stage shapes");
inline constexpr int P2_STAGES = 2;


// An operand shared by both lanes.  Written as one register twice (16-byte
// records, not records that hold each value twice) the packed instructions
// read it once.  They are bound by register reads: FFMA2 takes 3.3 cycles with
// three distinct pairs and 2.8 with one shared operand, two FFMA 2.0 but twice
// the issue slots (every mix of packed and scalar forms measured slower).  On
// the 786,432 x 65,536 cube a pass fell from 9.33 to 8.45 ms (6.5 cycles per
// pair and warp, 5 without any register conflict); the shared-memory traffic
// of the records halved.
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// r = c + x'.w of a point pair and one target record (w0, w1, w2, c)
template <int D>
__device__ __forceinline__ float2 pair_exponent(const float2 (&X)[3], float4 w) {
    float2 r = both(w.w);
    if (D == 3) r = __ffma2_rn(X[2], both(w.z), r);
    r = __ffma2_rn(X[1], both(w.y), r);
    return __ffma2_rn(X[0], both(w.x), r);
}

// Exact sub-tile for one point pair: maximum of r over the sub-tile, shift M
// raised to ceil(max) when the maximum exceeds it (rescaling the running sums
// by an exact power of two), then the sum of 2^(r - M).
template <int D>
__device__ __forceinline__ float2 lse_exact_subtile(const float4 *T, const float2 (&X)[3], float2 &M,
                                                    float2 &Sf, double2 &Sd) {
    float mx = -INFINITY, my = -INFINITY;
#pragma unroll 4
    for (int t = 0; t < P1_SUB; ++t) {
        const float2 r = pair_exponent<D>(X, T[t]);
        mx = fmaxf(mx, r.x);
        my = fmaxf(my, r.y);
    }
    if (mx > M.x) {
        const float mn = ceilf(mx), dl = M.x - mn;
        Sf.x *= pow2_int_f(dl);
        Sd.x *= pow2_int_d(dl);
        M.x = mn;
    }
    if (my > M.y) {
        const float mn = ceilf(my), dl = M.y - mn;
        Sf.y *= pow2_int_f(dl);
        Sd.y *= pow2_int_d(dl);
        M.y = mn;
    }
    const float2 nm = make_float2(-M.x, -M.y);
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int t = 0; t < P1_SUB; ++t) {
        const float2 r = pair_exponent<D>(X, T[t]);
        const float2 e = __fadd2_rn(r, nm);
        acc = __fadd2_rn(acc, make_float2(ex2_approx(e.x), ex2_approx(e.y)));
    }
    return acc;
}

// One staged tile of cnt <= P1_TS targets (the sub-tiles beyond hold padding, whose
// exponentials are 0) for PP point pairs: optimistic sub-tiles
// of P1_SUB targets with the running integral shift M, an exact sub-tile
// (raising M) when a sub-tile sum exceeds 2^60 or overflows.  One test covers
// the thread's point pairs (a test per pair cost 1 % of the pass).
template <int D, int PP>
__device__ __forceinline__ void lse_stage(const float4 *__restrict__ T, int cnt, const float2 (&X)[PP][3],
                                          float2 (&M)[PP], float2 (&Sf)[PP], double2 (&Sd)[PP]) {
#pragma unroll 1
    for (int t0 = 0; t0 < cnt; t0 += P1_SUB) {
        float2 acc0[PP], acc1[PP], nm[PP];
#pragma unroll
        for (int pp = 0; pp < PP; ++pp) nm[pp] = make_float2(-M[pp].x, -M[pp].y);
#pragma unroll
        for (int t = 0; t < P1_SUB; ++t) {
            const float4 w = T[t0 + t];
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
                const float2 e = __fadd2_rn(pair_exponent<D>(X[pp], w), nm[pp]);
                const float2 v = make_float2(ex2_approx(e.x), ex2_approx(e.y));
                if (t == 0) acc0[pp] = v;
                else if (t == 1) acc1[pp] = v;
                else if (t & 1) acc1[pp] = __fadd2_rn(acc1[pp], v);
                else acc0[pp] = __fadd2_rn(acc0[pp], v);
            }
        }
        float top = 0.0f;
#pragma unroll
        for (int pp = 0; pp < PP; ++pp) {
            acc0[pp] = __fadd2_rn(acc0[pp], acc1[pp]);
            top = max3f(top, acc0[pp].x, acc0[pp].y);
        }
        if (!(top <= P1_BIG)) {
#pragma unroll
            for (int pp = 0; pp < PP; ++pp)
                if (!(fmaxf(acc0[pp].x, acc0[pp].y) <= P1_BIG))
                    acc0[pp] = lse_exact_subtile<D>(T + t0, X[pp], M[pp], Sf[pp], Sd[pp]);
        }
#pragma unroll
        for (int pp = 0; pp < PP; ++pp) Sf[pp] = __fadd2_rn(Sf[pp], acc0[pp]);
    }
}

// One staged tile of cnt <= P2_TS point records (x0,x1,x2,u) for TPP
// target pairs held in registers: acc64 += sum over the tile of
// 2^(c_j + x'.w_j + u_q) = sum_q m_q p_qj, FP32 within the tile, FP64 across.
template <int D, int TPP>
__device__ __forceinline__ void grad_stage(const float4 *__restrict__ T, int cnt, const float2 (&W0)[TPP],
                                           const float2 (&W1)[TPP], const float2 (&W2)[TPP],
                                           const float2 (&C)[TPP], double2 (&acc64)[TPP]) {
    float2 acc[TPP];
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) acc[tp] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int i = 0; i < cnt; ++i) {
        const float4 p = T[i];
        const float2 x0 = both(p.x), x1 = both(p.y), x2 = both(p.z), u = both(p.w);
#pragma unroll
        for (int tp = 0; tp < TPP; ++tp) {
            float2 t = C[tp];
            if (D == 3) t = __ffma2_rn(x2, W2[tp], t);
            t = __ffma2_rn(x1, W1[tp], t);
            t = __ffma2_rn(x0, W0[tp], t);
            t = __fadd2_rn(t, u);
            acc[tp] = __fadd2_rn(acc[tp], make_float2(ex2_approx(t.x), ex2_approx(t.y)));
        }
    }
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) {
        acc64[tp].x += (double)acc[tp].x;
        acc64[tp].y += (double)acc[tp].y;
    }
}

// The same with the sums of the conditional centroids: cen[tp][k] += sum over the
// half stage of e x'_k, cen[tp][D] += sum of e, in FP32 per 256 points; acc runs on
// over the stage's two halves (whose first sum it is) as in grad_stage.
template <int D, int TPP, bool FIRST>
__device__ __forceinline__ void cent_half(const float4 *__restrict__ T, int cnt, const float2 (&W0)[TPP],
                                          const float2 (&W1)[TPP], const float2 (&W2)[TPP],
                                          const float2 (&C)[TPP], float2 (&acc)[TPP],
                                          double2 (&cen)[TPP][D + 1]) {
    float2 s[TPP], sx[TPP][D];
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) {
        s[tp] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < D; ++k) sx[tp][k] = make_float2(0.f, 0.f);
    }
#pragma unroll 4
    for (int i = 0; i < cnt; ++i) {
        const float4 p = T[i];
        const float2 x0 = both(p.x), x1 = both(p.y), x2 = both(p.z), u = both(p.w);
#pragma unroll
        for (int tp = 0; tp < TPP; ++tp) {
            float2 t = C[tp];
            if (D == 3) t = __ffma2_rn(x2, W2[tp], t);
            t = __ffma2_rn(x1, W1[tp], t);
            t = __ffma2_rn(x0, W0[tp], t);
            t = __fadd2_rn(t, u);
            const float2 e = make_float2(ex2_approx(t.x), ex2_approx(t.y));
            acc[tp] = __fadd2_rn(acc[tp], e);
            if (!FIRST) s[tp] = __fadd2_rn(s[tp], e);
            sx[tp][0] = __ffma2_rn(e, x0, sx[tp][0]);
            sx[tp][1] = __ffma2_rn(e, x1, sx[tp][1]);
            if (D == 3) sx[tp][2] = __ffma2_rn(e, x2, sx[tp][2]);
        }
    }
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) {
        const float2 a = FIRST ? acc[tp] : s[tp];
        cen[tp][D].x += a.x, cen[tp][D].y += a.y;
#pragma unroll
        for (int k = 0; k < D; ++k) cen[tp][k].x += sx[tp][k].x, cen[tp][k].y += sx[tp][k].y;
    }
}
template <int D, int TPP>
__device__ __forceinline__ void cent_stage(const float4 *__restrict__ T, int cnt, const float2 (&W0)[TPP],
                                           const float2 (&W1)[TPP], const float2 (&W2)[TPP],
                                           const float2 (&C)[TPP], double2 (&acc64)[TPP],
                                           double2 (&cen)[TPP][D + 1]) {
    constexpr int HALF = 256;   // points per FP32 sum of the centroids
    static_assert(P2_TS == 2 * HALF, "two halves per stage");
    float2 acc[TPP];
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) acc[tp] = make_float2(0.f, 0.f);
    cent_half<D, TPP, true>(T, min(cnt, HALF), W0, W1, W2, C, acc, cen);
    if (cnt > HALF) cent_half<D, TPP, false>(T + HALF, cnt - HALF, W0, W1, W2, C, acc, cen);
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) {
        acc64[tp].x += (double)acc[tp].x;
        acc64[tp].y += (double)acc[tp].y;
    }
}

// (double)v 2^k for an integer-valued k <= 0, by the bits of a normal v > 0 (the
// conversion and the product would each take the FP64 pipe); else as written
__device__ __forceinline__ double scaled_d(float v, float k) {
    const unsigned b = __float_as_uint(v);
    if (b - 0x00800000u >= 0x7f000000u || !(k >= -896.0f)) return (double)v * pow2_int_d(k);
    return __hiloint2double((int)((b >> 3) + (896u << 20)) + ((int)k << 20), (int)(b << 29));
}

// log2 of the sum of k1 pass-1 partials (M, S): S 2^M each.  The first eight loads are
// in flight together and held for the sum (a load after the other, twice, took
// half of the combining kernels: 61,206 points of a 61,206 x 5,003 problem: 18 -> 14 us, the FP64 logarithm is
// most of the rest).
template <class F>
__device__ __forceinline__ double merge_partials(int k1, F load) {
    constexpr int HELD = 8;
    float2 v[HELD];
    float mx = kPadC;
#pragma unroll
    for (int k = 0; k < HELD; ++k) v[k] = k < k1 ? load(k) : make_float2(kPadC, 0.f);
#pragma unroll
    for (int k = 0; k < HELD; ++k) mx = fmaxf(mx, v[k].x);
#pragma unroll 4
    for (int k = HELD; k < k1; ++k) mx = fmaxf(mx, load(k).x);
    double tot = 0.0;
#pragma unroll
    for (int k = 0; k < HELD; ++k)
        if (k < k1) tot += scaled_d(v[k].y, v[k].x - mx);
#pragma unroll 4
    for (int k = HELD; k < k1; ++k) {
        const float2 w = load(k);
        tot += scaled_d(w.y, w.x - mx);
    }
    return (double)mx + log2(tot);
}

}  // namespace rsot
