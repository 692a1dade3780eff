// Dense FP64 evaluation with fixed-point exponents.
//
// GB300 has 2 FP64 lanes per SM and clock against 128 FP32/integer lanes, and
// the FP64 passes of rsot_dense.cu spend 25 FP64 operations per pair and pass.
// Here a pair costs one: its exponent and the fraction of its exponential are
// 64-bit integers, and one fma adds the term in FP64.
//
// Log2 domain: t_qj = B_j - kappa |x_q - y_j|^2 with kappa = log2(e) / (2 eps),
// B_j = ((psi_j - psi_0)/eps + ln nu_j) log2(e).
//   * Coordinates are scaled by sqrt(kappa) 2^s and rounded to integers
//     X = h 2^31 + l (0 <= l < 2^31, h kept modulo 2^32), so a difference is
//     D = dh 2^31 + dl with two 32-bit subtractions and no carry, and
//     kappa d^2 = 2^-F ( sum dh^2 + (sum dh dl >> 30) ),  F = 2 s - 62,
//     up to the dropped sum dl^2 2^-62 < 3 units (its mean and the shift's half
//     unit, together close to 1, are added to the columns' constants).  F is at most 52 and falls by
//     two for every factor 4 of the largest exponent that occurs (FxPar), whose
//     FP64 rounding grows alike.
//   * The exponent n = kappa d^2 - C (C: the column's constant, 64-bit, modulo
//     2^(64-F)) gives 2^-n = 2^-I T[i] q: I its integer part, T[i] = 2^(-i/2048)
//     from the next 11 bits (table of FP64 values), and q = 2^-g, g < 2^-11, as
//     1 - z + z^2/2 (1 - c z), z = g ln 2, in 32-bit integer multiplications
//     (c is 1/3 less the value that centres the dropped z^4/24: error below
//     2^-54); its FP64 bits are those of 1.0 minus the integer 2^53 (1 - q).
//   * A pair is skipped when an FP32 estimate of its exponent (the record of
//     the mixed pass 1, error below E) shows that it cannot matter: in pass 1
//     below 2^(-60) / n of the point's sum, in pass 2 below 2^(-60) nu_j / sum m
//     of the point's mass; all skipped terms together change a sum by less than
//     2^-60 of it and a gradient entry by less than 2^-60 nu_j.  The wrapped
//     integers are only read for pairs that are not skipped, whose exponents
//     lie inside the range that FxPar allows.
// Error of an exponent: about 2^-F (F = 52: 2.2e-16) against about 2^-53 of the
// largest of kappa d^2, B_j in the FP64 passes.
//
// The estimate needs the points' approximate log-partition: the FP32 pass 1 of
// the mixed path runs first (about a tenth of the time).  Where the estimate
// could be off by more than 16 or the exponents need F < 46 the records kernel
// raises kErrRange64 and the caller runs the FP64 passes instead.
#include <math.h>

#include <algorithm>

#include "rsot_internal.cuh"
#include "rsot_exp64.cuh"

namespace rsot {

// integer operand record: (h0, l0, h1, l1), (h2, l2, -C low, -C high)
struct FxRec {
    int4 a, b;
};

namespace {

constexpr int FX_THREADS = 128;
constexpr int FX_TS = 128;        // columns per shared-memory tile
constexpr int FX_TAB = 2048;      // 2^(-i/2048)
constexpr int FX_FMAX = 52, FX_FMIN = 46;
constexpr double kNegl = 60.0;    // skipped terms lie below 2^-60 of what they are added to

__device__ __forceinline__ unsigned ordered_key(float f) {
    const unsigned b = __float_as_uint(f);
    return b & 0x80000000u ? ~b : b | 0x80000000u;   // monotone; 0 is below every float
}
__device__ __forceinline__ float from_key(unsigned k) {
    return __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k);
}

// block maximum into *key
__device__ __forceinline__ void block_max_key(float v, unsigned *key) {
    __shared__ float sh[32];
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = fmaxf(v, sh[w]);
        if (v > -INFINITY) atomicMax(key, ordered_key(v));
    }
}

// log2 of v > 0 as an integer and a fraction in [-1/2, 1/2]: the fraction's
// error is 2^-53, not 2^-53 of |log2 v|
__device__ __forceinline__ double log2_split(double v, int &e) {
    double m = frexp(v, &e);   // [1/2, 1)
    if (m < 0.70710678118654752) {
        m *= 2.0;
        --e;
    }
    return log2(m);
}

// B_j as an unevaluated sum of three: (psi_j - psi_0)/eps log2(e) in
// double-double plus log2 nu_j split into integer and fraction
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

// 2^F (hi + lo) modulo 2^64, |hi| < 2^52
__device__ __forceinline__ long long to_fixed(double hi, double lo, int F) {
    const double ip = rint(hi);
    const double f = (hi - ip) + lo;
    return (long long)((unsigned long long)(long long)ip << F) + llrint(ldexp(f, F));
}

__device__ __forceinline__ int2 fx_coord(double x, double c0, double c1, int s) {
    // x (c0 + c1) 2^s rounded to an integer modulo 2^63, as limbs of base 2^31
    const double p = x * c0;
    const double e = fma(x, c0, -p) + x * c1;
    const double ps = ldexp(p, s - 31);
    const double h = floor(ps);
    const long long v = (long long)((unsigned long long)(long long)h << 31) +
                        llrint(fma(ps - h, 2147483648.0, ldexp(e, s)));
    return make_int2((int)(v >> 31), (int)(v & 0x7fffffff));
}

}  // namespace

// ----------------------------------------------------------------------------
// Order of the target rows of pass 2: by cells of a 2^b grid in Morton order
// (counting sort, once per problem), so that a warp's targets are near each
// other and most of a far point's pairs are skipped by whole warps: at eps 1e-3
// (98,304 x 16,384) pass 2 takes 1.6 ms, 3.7 in the caller's order.  The order inside
// a cell is whatever the atomics give; a row's sum does not depend on it.
// ----------------------------------------------------------------------------
constexpr int SORT_CELLS = 4096;

__global__ void k_cell_count(const double *__restrict__ y64, int64_t n, int d, double half,
                             int *__restrict__ cell, int *__restrict__ count) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int bits = d == 3 ? 4 : 6;
    int id = 0;
    for (int t = 0; t < d; ++t) {
        const double u = half > 0.0 ? (y64[j * d + t] / half + 1.0) * 0.5 : 0.0;
        const int c = min(max((int)(u * (1 << bits)), 0), (1 << bits) - 1);
        for (int b = 0; b < bits; ++b) id |= ((c >> b) & 1) << (d * b + t);
    }
    cell[j] = id;
    atomicAdd(&count[id], 1);
}

// exclusive scan of the 4,096 counts (one block of 1,024 threads)
__global__ void k_cell_scan(int *__restrict__ count) {
    __shared__ int sh[1024];
    int v[4], sum = 0;
    for (int k = 0; k < 4; ++k) {
        v[k] = sum;
        sum += count[threadIdx.x * 4 + k];
    }
    sh[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int t = threadIdx.x >= o ? sh[threadIdx.x - o] : 0;
        __syncthreads();
        sh[threadIdx.x] += t;
        __syncthreads();
    }
    const int base = threadIdx.x ? sh[threadIdx.x - 1] : 0;
    for (int k = 0; k < 4; ++k) count[threadIdx.x * 4 + k] = base + v[k];
}

__global__ void k_cell_scatter(const int *__restrict__ cell, int64_t n, int64_t n_pad,
                               int *__restrict__ offset, int *__restrict__ perm) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n) perm[atomicAdd(&offset[cell[j]], 1)] = (int)j;
    else if (j < n_pad) perm[j] = (int)j;
}

// ----------------------------------------------------------------------------
// Per point: R_q from the FP32 pass 1 (log2 sum_j 2^(t_qj + kappa |x'_q|^2)),
// the float operands of both passes and the integral shift of pass 1; per
// target: the float operands.  The ranges that fix F go into the result block.
// ----------------------------------------------------------------------------
__global__ void k_fx_operands(const float2 *__restrict__ part, int k1, int64_t nq_pad, int64_t nq,
                              const float *__restrict__ xs, const double *__restrict__ x64, int d,
                              double kappa, const double *__restrict__ mass, double t1,
                              const double *__restrict__ psi, double eps,
                              const double *__restrict__ nu, double msum, int64_t n, int64_t n_pad,
                              const float4 *__restrict__ tquad, float4 *__restrict__ ptrow,
                              float4 *__restrict__ ptcol, int *__restrict__ ptshift,
                              float4 *__restrict__ tgrow, float4 *__restrict__ tgcol,
                              EvalResult *__restrict__ res) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float negt = -INFINITY, bmax = -INFINITY, babs = -INFINITY;
    if (i < nq_pad) {
        float4 row = make_float4(0.f, 0.f, 0.f, INFINITY), col = make_float4(0.f, 0.f, 0.f, kPadC);
        int sh = 0;
        if (i < nq) {
            float mx = kPadC;
            for (int k = 0; k < k1; ++k) mx = fmaxf(mx, part[(int64_t)k * nq_pad + i].x);
            float tot = 0.f;
            for (int k = 0; k < k1; ++k) {
                const float2 v = part[(int64_t)k * nq_pad + i];
                tot += v.y * pow2_int_f(v.x - mx);
            }
            const float R = mx + log2f(tot);
            float x[3] = {0.f, 0.f, 0.f};
            double r2 = 0.0;
            for (int t = 0; t < d; ++t) {
                x[t] = xs[t * nq_pad + i];
                r2 = fma(x64[i * d + t], x64[i * d + t], r2);
            }
            const double tq = (double)R - kappa * r2;
            sh = (int)rint(fmin(fmax(tq, -1.0e9), 1.0e9));
            negt = (float)-tq;
            row = make_float4(x[0], x[1], x[2], R - (float)t1);
            col = make_float4(x[0], x[1], x[2], mass[i] > 0.0 ? -R : kPadC);
        }
        ptrow[i] = row;
        ptcol[i] = col;
        ptshift[i] = sh;
    }
    if (i < n_pad) {
        const float4 r = tquad[i];
        float thr = INFINITY;
        if (i < n) {
            double bh, bl;
            target_B(psi[i], psi[0], eps, nu[i], bh, bl);
            bmax = (float)bh;
            babs = fabsf((float)bh);
            thr = (float)(log2(nu[i] / msum) - kNegl) - r.w;
        }
        tgrow[i] = make_float4(r.x, r.y, r.z, thr);
        tgcol[i] = r;
    }
    block_max_key(negt, &res->fx_key[0]);
    block_max_key(bmax, &res->fx_key[1]);
    block_max_key(babs, &res->fx_key[2]);
}

// Integer operands, the fraction bits F and the estimate's margin E from the
// ranges, and the table of 2^(-i/2048).
__global__ void k_fx_records(const double *__restrict__ x64, int64_t nq, int64_t nq_pad,
                             const double *__restrict__ y64, int64_t n, int64_t n_pad, int d,
                             double c0, double c1, double kappa_diam2, double tmax,
                             const double *__restrict__ psi, double eps,
                             const double *__restrict__ nu, FxRec *__restrict__ prec,
                             FxRec *__restrict__ trec, int *__restrict__ tgshift,
                             double *__restrict__ tgscale, double *__restrict__ tab,
                             EvalResult *__restrict__ res) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double negt = from_key(res->fx_key[0]), bmax = from_key(res->fx_key[1]);
    const double babs = from_key(res->fx_key[2]);
    // |estimate - exponent| <= 7 roundings of 2^-24 of the terms' magnitudes
    const double E = 0x1p-20 * (babs + kappa_diam2);
    const double L = (bmax + negt + tmax + 4.0 * E + 4.0) / 0.9;   // largest kappa d^2 of a kept pair
    int F = FX_FMAX;
    while (F >= FX_FMIN && L >= ldexp(1.0, 62 - F)) F -= 2;
    const bool bad = F < FX_FMIN || !(E <= 16.0) || !(L > 0.0);
    if (bad) F = FX_FMIN;
    if (i == 0) {
        res->fx_F = F;
        res->fx_E = (float)E;
        if (bad) atomicOr(&res->flags, kErrRange64);
    }
    const int s = (F + 62) / 2;
    if (bad) return;
    if (i < nq_pad) {
        int2 c[3] = {};
        if (i < nq)
            for (int t = 0; t < d; ++t) c[t] = fx_coord(x64[i * d + t], c0, c1, s);
        FxRec r;
        r.a = make_int4(c[0].x, c[0].y, c[1].x, c[1].y);
        r.b = make_int4(c[2].x, c[2].y, 0, 0);
        prec[i] = r;
    }
    if (i < n_pad) {
        int2 c[3] = {};
        long long C = 0;
        int sh = 0;
        double scale = 0.0;
        if (i < n) {
            for (int t = 0; t < d; ++t) c[t] = fx_coord(y64[i * d + t], c0, c1, s);
            double bh, bl;
            target_B(psi[i], psi[0], eps, nu[i], bh, bl);
            C = 1 - to_fixed(bh, bl, F);
            const double fl = rint(bh);
            sh = (int)fl;
            scale = exp2((bh - fl) + bl);
        }
        FxRec r;
        r.a = make_int4(c[0].x, c[0].y, c[1].x, c[1].y);
        r.b = make_int4(c[2].x, c[2].y, (int)(C & 0xffffffffll), (int)(C >> 32));
        trec[i] = r;
        tgshift[i] = sh;
        tgscale[i] = scale;
    }
    if (i < FX_TAB) {
        // 2^(-i/2048) = 2^(j/64) e^r / 2 with 2048 - i = 32 j + 2048 r / ln 2
        const int m = FX_TAB - (int)i, j = m >> 5;
        const double r = (double)(m & 31) * (kLn2 / 2048.0);
        double p = 1.0 / 40320.0;
        p = fma(p, r, 1.0 / 5040.0);
        p = fma(p, r, 1.0 / 720.0);
        p = fma(p, r, 1.0 / 120.0);
        p = fma(p, r, 1.0 / 24.0);
        p = fma(p, r, 1.0 / 6.0);
        p = fma(p, r, 0.5);
        p = fma(p, r, 1.0) * r;
        const double2 h = j < 64 ? kExp2Tab[j] : make_double2(2.0, 0.0);
        tab[i] = 0.5 * (fma(h.x, p, h.y) + h.x);
    }
}

// ----------------------------------------------------------------------------
// One pass: out[chunk][row] = sum over the chunk's columns of
// 2^(C_col - kappa d^2 - shift_row).  Pass 1: rows = points, columns = targets;
// pass 2: rows = targets (in the order of perm), columns = points.
// ----------------------------------------------------------------------------
template <int D, int R>
__global__ void __launch_bounds__(FX_THREADS)
    k_fx_pass(const FxRec *__restrict__ rowrec, const float4 *__restrict__ rowf,
              const int *__restrict__ rowshift, int neg_shift, const int *__restrict__ perm,
              int64_t rows_pad,
              const FxRec *__restrict__ colrec, const float4 *__restrict__ colf, int64_t cols,
              int64_t chunk, const double *__restrict__ tab, double *__restrict__ out,
              const EvalResult *__restrict__ res) {
    if (res->flags & kErrRange64) return;
    __shared__ __align__(16) FxRec s_rec[FX_TS];
    __shared__ __align__(16) float4 s_f[FX_TS];
    __shared__ double s_tab[FX_TAB];
    const int tid = threadIdx.x;
    for (int i = tid; i < FX_TAB / 2; i += FX_THREADS)
        reinterpret_cast<double2 *>(s_tab)[i] = reinterpret_cast<const double2 *>(tab)[i];
    const int F = res->fx_F;
    const float E = res->fx_E;
    const int shE = F - 32, shI = F - 46, shG = 75 - F;
    int H[R][3], Lo[R][3], rs[R], at[R];
    float4 xf[R];
    double acc[R];
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int64_t i = (int64_t)blockIdx.x * (FX_THREADS * R) + k * FX_THREADS + tid;
        acc[k] = 0.0;
        xf[k] = make_float4(0.f, 0.f, 0.f, INFINITY);
        rs[k] = 0;
        FxRec r;
        r.a = r.b = make_int4(0, 0, 0, 0);
        at[k] = -1;
        if (i < rows_pad) {
            at[k] = perm ? perm[i] : (int)i;
            r = rowrec[at[k]];
            xf[k] = rowf[at[k]];
            xf[k].w -= 2.0f * E;
            rs[k] = rowshift[at[k]];
            if (neg_shift) rs[k] = -rs[k];
            rs[k] = (int)((unsigned)rs[k] << shE);
        }
        H[k][0] = r.a.x, Lo[k][0] = r.a.y;
        H[k][1] = r.a.z, Lo[k][1] = r.a.w;
        H[k][2] = r.b.x, Lo[k][2] = r.b.y;
    }
    const int64_t c_begin = (int64_t)blockIdx.y * chunk;
    const int64_t c_end = min(cols, c_begin + chunk);
    for (int64_t t0 = c_begin; t0 < c_end; t0 += FX_TS) {
        const int cnt = (int)min((int64_t)FX_TS, c_end - t0);
        __syncthreads();
        if (tid < cnt) {
            s_rec[tid] = colrec[t0 + tid];
            s_f[tid] = colf[t0 + tid];
        }
        __syncthreads();
        for (int c = 0; c < cnt; ++c) {
            const float4 f = s_f[c];
            const int4 a = s_rec[c].a, b = s_rec[c].b;
            const long long nc = (long long)(((unsigned long long)(unsigned)b.w << 32) | (unsigned)b.z);
#pragma unroll
            for (int k = 0; k < R; ++k) {
                float e = f.w;
                if (D == 3) e = fmaf(f.z, xf[k].z, e);
                e = fmaf(f.x, xf[k].x, fmaf(f.y, xf[k].y, e));
                if (e >= xf[k].w) {
                    const int h0 = H[k][0] - a.x, h1 = H[k][1] - a.z;
                    const int l0 = Lo[k][0] - a.y, l1 = Lo[k][1] - a.w;
                    long long hh = (long long)h0 * h0 + nc;
                    long long mid = (long long)h0 * l0;
                    hh += (long long)h1 * h1;
                    mid += (long long)h1 * l1;
                    if (D == 3) {
                        const int h2 = H[k][2] - b.x, l2 = Lo[k][2] - b.y;
                        hh += (long long)h2 * h2;
                        mid += (long long)h2 * l2;
                    }
                    hh += mid >> 30;
                    const unsigned lo = (unsigned)hh;
                    const int hi = (int)(hh >> 32) + rs[k];
                    const int ex = hi >> shE;                       // integer part
                    const unsigned off = ((unsigned)hi >> shI) & ((FX_TAB - 1u) << 3);
                    const double T = *reinterpret_cast<const double *>(
                        reinterpret_cast<const char *>(s_tab) + off);
                    const unsigned G = __funnelshift_l(lo, (unsigned)hi, shG);   // g 2^43
                    const unsigned Gl = lo << shG;
                    // z = g ln 2 in units of 2^-75 (2^21: rounds the shift below)
                    constexpr unsigned kL1 = 0xB17217F7u, kL2 = 0xD1CF79ABu;
                    unsigned long long z = (unsigned long long)G * kL1 + (1u << 21);
                    z += __umulhi(G, kL2);
                    z += __umulhi(Gl, kL1);
                    const unsigned zh = (unsigned)(z >> 32);                     // 2^-43
                    const unsigned s2 = __umulhi(zh, zh);                        // 2^-54
                    const unsigned y = zh - __umulhi(s2, 698996u);
                    z -= (unsigned long long)__umulhi(zh, y) << 20;
                    const double q = __longlong_as_double(0x3FF0000000000000ll - (long long)(z >> 22));
                    const double Ts = __hiloint2double(__double2hiint(T) - (ex << 20), __double2loint(T));
                    acc[k] = fma(Ts, q, acc[k]);
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < R; ++k)
        if (at[k] >= 0) out[(int64_t)blockIdx.y * rows_pad + at[k]] = acc[k];
}

// Per point: L_q, the mass's J term, and the column constant of pass 2,
// u_q = log2(m_q / S_q) - shift_q.
__global__ void k_fx_combine(const double *__restrict__ part, int k1, int64_t nq, int64_t nq_pad,
                             const int *__restrict__ shift, const double *__restrict__ mass,
                             const double *__restrict__ psi, double eps, FxRec *__restrict__ prec,
                             double *__restrict__ lse_buf, double *__restrict__ blockJ,
                             const EvalResult *__restrict__ res) {
    __shared__ double sh[32];
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double contrib = 0.0;
    if (res->flags & kErrRange64) return;
    if (q < nq) {
        double S = 0.0;
        for (int k = 0; k < k1; ++k) S += part[(int64_t)k * nq_pad + q];
        const int M = shift[q];
        const double L = fma((double)M, kLn2, log(S));
        lse_buf[q] = L;
        const double m = mass[q];
        if (m > 0.0) {
            contrib = m * (psi[0] + eps * L);
            int em, es;
            const double fm = log2_split(m, em), fs = log2_split(S, es);
            const long long C = 1 - to_fixed((double)(em - es - M), fm - fs, res->fx_F);
            prec[q].b.z = (int)(C & 0xffffffffll);
            prec[q].b.w = (int)(C >> 32);
        }
    }
    const double s = block_sum_d(contrib, sh);
    if (threadIdx.x == 0) blockJ[blockIdx.x] = s;
}

__global__ void k_fx_grad(const double *__restrict__ part2, int s2, int64_t stride,
                          const double *__restrict__ scale, const double *__restrict__ nu, int64_t n,
                          double *__restrict__ grad) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double g = 0.0;
    for (int s = 0; s < s2; ++s) g += part2[(int64_t)s * stride + j];
    grad[j] = fma(g, scale[j], -nu[j]);
}

// ----------------------------------------------------------------------------
namespace {

int fx_split(int64_t units, int64_t tiles, int64_t slots) {
    // the smallest split that fills the slots (a multiple of a wave within 5 %)
    int best = 1;
    double best_eff = 0.0;
    for (int64_t s = 1; s <= std::min<int64_t>(tiles, 256); ++s) {
        const int64_t items = units * s, waves = (items + slots - 1) / slots;
        const double eff = (double)items / (double)(waves * slots);
        if (eff > best_eff + 0.01) best_eff = eff, best = (int)s;
        if (items >= slots && eff >= 0.95) return (int)s;
    }
    return best;
}

// rows per thread: 2 share a column's loads, 1 where that leaves SMs idle
inline int fx_rows(const rsot_problem *p, int64_t rows, int64_t cols) {
    return rows / (2 * FX_THREADS) * (cols / (4 * FX_TS)) >= 5 * p->num_sms ? 2 : 1;
}

template <int D>
void fx_launch(rsot_problem *p, int R, const FxRec *rr, const float4 *rf, const int *rsh, int neg, const int *perm,
               int64_t rows, int64_t rows_pad, const FxRec *cr, const float4 *cf, int64_t cols, int64_t chunk, int splits,
               double *out) {
    // rows_pad is the stride of out; blocks of padding rows alone are not launched
    dim3 g((unsigned)((rows + FX_THREADS * R - 1) / (FX_THREADS * R)), (unsigned)splits);
    if (R == 2)
        k_fx_pass<D, 2><<<g, FX_THREADS, 0, p->stream>>>(rr, rf, rsh, neg, perm, rows_pad, cr, cf, cols, chunk,
                                                         p->fx_tab, out, p->res_dev);
    else
        k_fx_pass<D, 1><<<g, FX_THREADS, 0, p->stream>>>(rr, rf, rsh, neg, perm, rows_pad, cr, cf, cols, chunk,
                                                         p->fx_tab, out, p->res_dev);
}

}  // namespace

void fx64_free(rsot_problem *p) {
    cudaFree(p->fx_buf);
    p->fx_buf = nullptr;
}

// buffers of the fixed-point passes, once per problem; false: no memory (the
// FP64 passes need none of them)
static bool fx_alloc(rsot_problem *p) {
    if (p->fx_buf) return true;
    const int64_t slots = (int64_t)p->num_sms * 5;
    const int64_t b1 = FX_THREADS * fx_rows(p, p->nq, p->n), b2 = FX_THREADS * fx_rows(p, p->n, p->nq);
    auto chunked = [&](int64_t rows, int64_t blk, int64_t cols, int &split, int64_t &chunk) {
        const int64_t tiles = (cols + FX_TS - 1) / FX_TS;
        split = fx_split((rows + blk - 1) / blk, tiles, slots);
        chunk = (tiles + split - 1) / split * FX_TS;
        split = (int)((cols + chunk - 1) / chunk);
    };
    chunked(p->nq, b1, p->n, p->fx_k1, p->fx_chunk1);
    chunked(p->n, b2, p->nq, p->fx_s2, p->fx_chunk2);
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t np = (size_t)p->nq_pad, nt = (size_t)p->n_pad;
    const size_t o_prec = take(np * sizeof(FxRec)), o_trec = take(nt * sizeof(FxRec));
    const size_t o_prow = take(np * 16), o_pcol = take(np * 16), o_psh = take(np * 4);
    const size_t o_trow = take(nt * 16), o_tcol = take(nt * 16), o_tsh = take(nt * 4);
    const size_t o_tsc = take(nt * 8), o_tab = take(FX_TAB * 8);
    const size_t o_perm = take(nt * 4), o_cell = take(nt * 4 + SORT_CELLS * 4);
    const size_t o_p1 = take(np * 8 * p->fx_k1), o_p2 = take(nt * 8 * p->fx_s2);
    char *b = nullptr;
    if (cudaMalloc(&b, at) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    p->fx_buf = b;
    p->fx_prec = reinterpret_cast<FxRec *>(b + o_prec);
    p->fx_trec = reinterpret_cast<FxRec *>(b + o_trec);
    p->fx_ptrow = reinterpret_cast<float4 *>(b + o_prow);
    p->fx_ptcol = reinterpret_cast<float4 *>(b + o_pcol);
    p->fx_ptshift = reinterpret_cast<int *>(b + o_psh);
    p->fx_tgrow = reinterpret_cast<float4 *>(b + o_trow);
    p->fx_tgcol = reinterpret_cast<float4 *>(b + o_tcol);
    p->fx_tgshift = reinterpret_cast<int *>(b + o_tsh);
    p->fx_tgscale = reinterpret_cast<double *>(b + o_tsc);
    p->fx_tab = reinterpret_cast<double *>(b + o_tab);
    p->fx_part1 = reinterpret_cast<double *>(b + o_p1);
    p->fx_part2 = reinterpret_cast<double *>(b + o_p2);
    p->fx_perm = reinterpret_cast<int *>(b + o_perm);
    int *cell = reinterpret_cast<int *>(b + o_cell), *count = cell + nt;
    cudaMemsetAsync(count, 0, SORT_CELLS * 4, p->stream);
    const unsigned nb = (unsigned)((p->n_pad + 255) / 256);
    k_cell_count<<<nb, 256, 0, p->stream>>>(p->y64, p->n, p->d, p->half_ext, cell, count);
    k_cell_scan<<<1, 1024, 0, p->stream>>>(count);
    k_cell_scatter<<<nb, 256, 0, p->stream>>>(cell, p->n, p->n_pad, count, p->fx_perm);
    // once per problem: a later evaluation may run on another stream
    if (cudaStreamSynchronize(p->stream) != cudaSuccess) {
        cudaGetLastError();
        fx64_free(p);
        return false;
    }
    return true;
}

bool fx64_ready(rsot_problem *p, double eps) {
    const double kappa = kLog2e / (2.0 * eps);
    // the estimate's error bound must allow a decision (see k_fx_records)
    if (!(kappa * p->diam2 <= 0x1p23) || !(p->msum > 0.0)) return false;
    return fx_alloc(p);
}

// the FP32 estimate of R_q and of the exponents' ranges: terms below 2^-t1 of a
// point's sum (pass 1) and below 2^-60 nu_j / sum m (pass 2) are told apart
cudaError_t launch_estimate(rsot_problem *p, const double *psi, double eps, double t1) {
    cudaStream_t st = p->stream;
    const double kappa = kLog2e / (2.0 * eps);
    cudaError_t e = launch_mixed_pass1(p, psi, eps);
    if (e) return e;
    const unsigned nb = (unsigned)((std::max(p->nq_pad, p->n_pad) + 255) / 256);
    trace_begin(p, "fx_operands");
    k_fx_operands<<<nb, 256, 0, st>>>(p->part1, p->k1, p->nq_pad, p->nq, p->xs, p->x64, p->d, kappa,
                                      p->mass, t1, psi, eps, p->nu, p->msum, p->n, p->n_pad, p->tquad,
                                      p->fx_ptrow, p->fx_ptcol, p->fx_ptshift, p->fx_tgrow,
                                      p->fx_tgcol, p->res_dev);
    trace_end(p);
    return cudaGetLastError();
}

cudaError_t launch_dense_fx64(rsot_problem *p, const double *psi, double eps, double *grad) {
    cudaStream_t st = p->stream;
    const double kappa = kLog2e / (2.0 * eps);
    // sqrt(kappa) as c0 + c1: kappa = (1/eps) log2(e) / 2 in double-double
    const double inv = 1.0 / eps, inv_lo = -fma(inv, eps, -1.0) / eps;
    const double kh = inv * (0.5 * kLog2e);
    const double kl = fma(inv, 0.5 * kLog2e, -kh) + inv * (0.5 * 2.0355273740931033e-17) +
                      inv_lo * (0.5 * kLog2e);
    const double c0 = sqrt(kh), c1 = (-fma(c0, c0, -kh) + kl) / (2.0 * c0);
    const double t1 = kNegl + log2((double)p->n) + 1.0;
    const double tmax = std::max(t1, kNegl + log2(p->msum / p->nu_min));
    cudaError_t e = launch_estimate(p, psi, eps, t1);
    if (e) return e;
    const unsigned nb = (unsigned)((std::max(p->nq_pad, p->n_pad) + 255) / 256);
    trace_begin(p, "fx_records");
    k_fx_records<<<std::max(nb, (unsigned)(FX_TAB / 256)), 256, 0, st>>>(
        p->x64, p->nq, p->nq_pad, p->y64, p->n, p->n_pad, p->d, c0, c1, kappa * p->diam2, tmax, psi,
        eps, p->nu, p->fx_prec, p->fx_trec, p->fx_tgshift, p->fx_tgscale, p->fx_tab, p->res_dev);
    trace_end(p);
    trace_begin(p, "fx_lse");
    const int r1 = fx_rows(p, p->nq, p->n), r2 = fx_rows(p, p->n, p->nq);
    (p->d == 3 ? fx_launch<3> : fx_launch<2>)(p, r1, p->fx_prec, p->fx_ptrow, p->fx_ptshift, 0, nullptr, p->nq, p->nq_pad,
                                              p->fx_trec, p->fx_tgcol, p->n, p->fx_chunk1, p->fx_k1,
                                              p->fx_part1);
    trace_end(p);
    trace_begin(p, "fx_combine");
    const int nbq = (int)((p->nq_pad + 255) / 256);
    k_fx_combine<<<nbq, 256, 0, st>>>(p->fx_part1, p->fx_k1, p->nq, p->nq_pad, p->fx_ptshift, p->mass,
                                      psi, eps, p->fx_prec, p->lse_buf, p->blockJ, p->res_dev);
    trace_end(p);
    trace_begin(p, "fx_grad");
    (p->d == 3 ? fx_launch<3> : fx_launch<2>)(p, r2, p->fx_trec, p->fx_tgrow, p->fx_tgshift, 1, p->fx_perm, p->n, p->n_pad,
                                              p->fx_prec, p->fx_ptcol, p->nq, p->fx_chunk2, p->fx_s2,
                                              p->fx_part2);
    trace_end(p);
    trace_begin(p, "finalize_grad");
    k_fx_grad<<<(unsigned)((p->n + 255) / 256), 256, 0, st>>>(p->fx_part2, p->fx_s2, p->n_pad,
                                                              p->fx_tgscale, p->nu, p->n, grad);
    trace_end(p);
    return launch_finalize_J64(p, psi, eps, nbq);
}

}  // namespace rsot
