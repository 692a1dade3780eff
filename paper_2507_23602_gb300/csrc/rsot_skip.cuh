// Skipping of pairs that cannot matter, for the dense FP64 (rsot_fx64.cu) and
// compensated (rsot_cx.cu) passes; the operands are prepared in rsot_skip.cu.
//
// With k = log2(e)/(2 eps), r_qj = c_j + x'_q.w_j the mixed pass's FP32 exponent
// and t_qj = r_qj - k |x'_q|^2 = B_j - k |x'_q - y'_j|^2, a pair is needed
//   pass 1: when r_qj >= max_j r_qj - t1, t1 = 60 + log2(n) + 1 (what is dropped
//           stays below 2^-60 of the point's sum);
//   pass 2: when r_qj - R_q >= log2(nu_j / sum m) - 60 (what is dropped stays
//           below 2^-60 nu_j of the target's mass).
// Both tests carry the margin 2 E, E = 2^-20 (max |B_j| + k diam^2): seven
// roundings of 2^-24 of the terms' magnitudes bound the FP32 exponent's error.
// A warp first tests 32 columns at a time, one per lane, against the ball of
// its own rows (a column's value B_j or A_q = k |x'_q|^2 - R_q plus the rows'
// largest against k dist^2), then each pair of the columns that remain.  The
// pair test alone (3 FMA, compare, vote) took half of a pass at eps = 1e-3 on
// 98,304 x 65,536.
#pragma once

#include "rsot_internal.cuh"

namespace rsot {

// The warp's rows: centre and radius of their box, largest value plus slack.
struct RowBall {
    float c0, c1, c2, r, top;
};

__device__ __forceinline__ float warp_max_f(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// two rows of this lane: positions (times scale) and values; value -inf: no row
__device__ __forceinline__ RowBall row_ball(float4 a, float va, float4 b, float vb, float scale) {
    RowBall w;
    w.top = warp_max_f(fmaxf(va, vb));
    const bool ia = va > -INFINITY, ib = vb > -INFINITY;
    const float xa[3] = {a.x, a.y, a.z}, xb[3] = {b.x, b.y, b.z};
    float c[3], r2 = 0.f;
    for (int t = 0; t < 3; ++t) {
        const float hi = warp_max_f(fmaxf(ia ? xa[t] : -INFINITY, ib ? xb[t] : -INFINITY)) * scale;
        const float lo = -warp_max_f(fmaxf(ia ? -xa[t] : -INFINITY, ib ? -xb[t] : -INFINITY)) * scale;
        c[t] = 0.5f * (hi + lo);
        r2 = fmaf(0.25f * (hi - lo), hi - lo, r2);
    }
    w.c0 = c[0], w.c1 = c[1], w.c2 = c[2];
    w.r = sqrtf(r2) * 1.0001f;
    return w;
}

// this lane's column (position times scale, value) against the warp's rows
__device__ __forceinline__ bool ball_needs(const RowBall &w, float4 col, float value, float scale, float k) {
    const float d0 = fmaf(-col.x, scale, w.c0), d1 = fmaf(-col.y, scale, w.c1), d2 = fmaf(-col.z, scale, w.c2);
    const float d = sqrt_sfu(fmaf(d0, d0, fmaf(d1, d1, d2 * d2)));
    const float near = fmaxf(d * 0.9999f - w.r, 0.f);
    return value + w.top >= near * near * k;
}

// the estimate's error bound E of the evaluation
__device__ __forceinline__ float skip_error(const EvalResult *res, float kdiam2) {
    return 0x1p-20f * (from_key(res->fx_key[2]) + kdiam2);
}

// B_j = ((psi_j - psi_0)/eps + ln nu_j) log2(e) as hi + lo, beyond FP64; and the
// split log2 of v > 0 into an integer and a fraction in [-1/2, 1/2] (whose
// error is 2^-53, not 2^-53 of |log2 v|)
__device__ __forceinline__ double log2_split(double v, int &e) {
    double m = frexp(v, &e);   // [1/2, 1)
    if (m < 0.70710678118654752) {
        m *= 2.0;
        --e;
    }
    return log2(m);
}

__device__ __forceinline__ void target_B(double ps, double psic, double eps, double nu, double &hi,
                                         double &lo) {
    constexpr double kL2eH = 1.4426950408889634, kL2eL = 2.0355273740931033e-17;
    const double s = ps - psic, bb = s - ps;
    const double se = (ps - (s - bb)) - (psic + bb);           // s + se = ps - psic exactly
    const double q = s / eps;
    const double qe = (fma(-q, eps, s) + se) / eps;
    const double p = q * kL2eH;
    const double pe = fma(q, kL2eH, -p) + fma(q, kL2eL, qe * kL2eH);
    int e;
    const double f = log2_split(nu, e);
    const double a = p + (double)e, ab = a - p;
    hi = a;
    lo = ((p - (a - ab)) + ((double)e - ab)) + pe + f;
}

// The warp's rows: their box in the columns' units (centre and half edges, 2k or 1
// times positions) and the factor of the distance.
struct Box {
    float c[3], h[3], f;
};

// this lane's column at (x, y, z): value - k dist^2
template <int D>
__device__ __forceinline__ float box_bound(const Box &b, float4 col, float value) {
    const float x[3] = {col.x, col.y, col.z};
    float d2 = 0.f;
#pragma unroll
    for (int t = 0; t < D; ++t) {
        const float d = fmaxf(fabsf(x[t] - b.c[t]) - b.h[t], 0.f);
        d2 = fmaf(d, d, d2);
    }
    return fmaf(-d2, b.f, value);
}

// box of the warp's rows, lo and hi per lane; widened for the rounding of both sides
template <int D>
__device__ __forceinline__ Box make_box(const float (&lo)[3], const float (&hi)[3], float scale, float f) {
    Box b;
    b.f = f * 0.9999f;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
        const float H = t < D ? warp_max_f(hi[t]) : 0.f, L = t < D ? -warp_max_f(-lo[t]) : 0.f;
        b.c[t] = 0.5f * (H + L) * scale;
        b.h[t] = (0.5f * (H - L) + 1e-6f * (fabsf(H) + fabsf(L))) * scale;
    }
    return b;
}

}  // namespace rsot
