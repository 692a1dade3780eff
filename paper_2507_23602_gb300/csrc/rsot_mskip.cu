// Dense mixed evaluations outside the solver: the passes of rsot_dense.cu without
// the pairs that cannot change a sum.
//
// In the unit cube at eps = 1e-3 a term falls below 2^-60 of its sum within a third
// of the edge, so four pairs of five add nothing.  The sums here keep every term
// that can matter, and its FP32 arithmetic, grouping and order (the shifts M, the
// sub-tiles of 16 targets and stages of 512 are those of lse_stage and grad_stage),
// so the results are those of the dense passes to 2^-60 of a sum.  The solver's
// evaluations stay with the dense passes bit by bit: its iterates follow the last
// bit of a sum (rsot_solve.cpp).
//
// A warp holds 64 PP neighbouring rows (points in pass 1, targets in pass 2, in the
// order of a cell grid's Morton curve) and takes the columns in their own order, 32
// at a time: each lane tests one against the box of the warp's rows, then the warp
// runs over the columns that remain.  With k = log2(e)/(2 eps) and the exponent
// t_qj = B_j - k |x_q - y_j|^2 + A_q (A_q = k |x_q|^2 in pass 1, + u_q in pass 2):
//   pass 1 needs j when B_j - k dist^2 + max_q (k |x_q|^2 - log2 S_q) >= -t1, S_q the
//     point's sum so far and t1 = 61 + log2 n: all that is dropped stays below 2^-60
//     of the sum (nothing is dropped before a point has its first sub-tile, and a
//     dropped term could not have raised M);
//   pass 2 needs q when A_q - k dist^2 + max_j (B_j - log2 nu_j) >= -(61 + log2 nq):
//     what is dropped stays below 2^-60 nu_j.
// Both tests carry a margin of 2^-19 (|terms|), twice the bound of the FP32
// exponents' error (rsot_skip.cuh).
// Bound: the packed FP32 instructions of the pairs that remain, and about ten
// instructions a column for the loop over a mask's bits (shared by 128 rows).
// 786,432 x 65,536, eps 1e-3: 8.4 -> 3.4 and 8.5 -> 3.4 ms, the call 17.0 -> 7.05.
#include <math.h>

#include <algorithm>

#include "rsot_internal.cuh"
#include "rsot_inner.cuh"
#include "rsot_skip.cuh"

namespace rsot {
namespace {

constexpr int MS_WARPS = 4, MS_THREADS = 32 * MS_WARPS;

template <int D, int PP>
__global__ void __launch_bounds__(MS_THREADS, 8)
    k_lse_skip(const float *__restrict__ xs, const int *__restrict__ perm, int64_t nq, int64_t nq_pad,
               const float4 *__restrict__ tquad, int n, int chunk, float k, float kdiam2, float t1,
               float2 *__restrict__ part) {
    pdl_enter();
    __shared__ __align__(16) float4 s_t[MS_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *const T = s_t[warp];
    const int64_t i0 = ((int64_t)blockIdx.x * MS_WARPS + warp) * (32 * PP);   // point pairs
    if (2 * i0 >= nq) return;
    int q[PP];
    const int kc = blockIdx.y, t_begin = kc * chunk, t_end = min(n, t_begin + chunk);
    const float inv4k = 0.25f / k;
    float2 X[PP][3], M[PP], Sf[PP];
    double2 Sd[PP];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int pp = 0; pp < PP; ++pp) {
        q[pp] = 2 * perm[i0 + 32 * pp + lane];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            X[pp][t] = t < D ? *reinterpret_cast<const float2 *>(xs + t * nq_pad + q[pp]) : make_float2(0.f, 0.f);
            if (q[pp] < nq) lo[t] = fminf(lo[t], X[pp][t].x), hi[t] = fmaxf(hi[t], X[pp][t].x);
            if (q[pp] + 1 < nq) lo[t] = fminf(lo[t], X[pp][t].y), hi[t] = fmaxf(hi[t], X[pp][t].y);
        }
        M[pp] = make_float2(kPadC, kPadC);
        Sf[pp] = make_float2(0.f, 0.f);
        Sd[pp] = make_double2(0.0, 0.0);
    }
    // columns in units of w = 2k y'
    const Box box = make_box<D>(lo, hi, 2.f * k, inv4k);
    float thr = -INFINITY;
    const auto load = [&](int g) { return g + lane < t_end ? tquad[g + lane] : make_float4(0.f, 0.f, 0.f, kPadC); };
    float4 nxt = load(t_begin);
#pragma unroll 1
    for (int g = t_begin; g < t_end; g += 32) {
        const float4 w = nxt;
        nxt = load(g + 32);
        __syncwarp();
        T[lane] = w;
        const float B = fmaf(fmaf(w.x, w.x, fmaf(w.y, w.y, w.z * w.z)), inv4k, w.w);
        const float bound = box_bound<D>(box, w, B) + 0x1p-19f * (fabsf(B) + kdiam2);
        const unsigned need = __ballot_sync(0xffffffffu, bound >= thr);
        __syncwarp();
#pragma unroll 1
        for (int t0 = 0; t0 < 32; t0 += P1_SUB) {
            const unsigned m = (need >> t0) & 0xffffu;
            if (!m) continue;
            float2 acc0[PP], acc1[PP], nm[PP];
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
                nm[pp] = make_float2(-M[pp].x, -M[pp].y);
                acc0[pp] = acc1[pp] = make_float2(0.f, 0.f);
            }
            // even and odd targets have their own sums, as in lse_stage
            const auto add = [&](float2 (&acc)[PP], const float4 v) {
#pragma unroll
                for (int pp = 0; pp < PP; ++pp) {
                    const float2 e = __fadd2_rn(pair_exponent<D>(X[pp], v), nm[pp]);
                    acc[pp] = __fadd2_rn(acc[pp], make_float2(ex2_approx(e.x), ex2_approx(e.y)));
                }
            };
            if (m == 0xffffu) {
#pragma unroll
                for (int t = 0; t < P1_SUB; t += 2) {
                    add(acc0, T[t0 + t]);
                    add(acc1, T[t0 + t + 1]);
                }
            } else {
#pragma unroll 1
                for (unsigned b = m & 0x5555u; b; b &= b - 1) add(acc0, T[t0 + __ffs(b) - 1]);
#pragma unroll 1
                for (unsigned b = m & 0xaaaau; b; b &= b - 1) add(acc1, T[t0 + __ffs(b) - 1]);
            }
            float top = 0.0f;
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
                acc0[pp] = __fadd2_rn(acc0[pp], acc1[pp]);
                top = fmaxf(top, fmaxf(acc0[pp].x, acc0[pp].y));
                if (!(acc0[pp].x + acc0[pp].y <= 2.f * P1_BIG)) top = INFINITY;   // NaN as well
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
        const bool stage_end = (g - t_begin + 32) % P1_TS == 0;
        if (stage_end || g - t_begin < P1_TS) {
            // the rows' largest k |x|^2 - log2 S (S from below by its exponent), after
            // every 32 targets of the first stage and after each later stage
            float V = -INFINITY;
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float S = (float)(h ? Sd[pp].y : Sd[pp].x) + (h ? Sf[pp].y : Sf[pp].x);
                    float r2 = 0.f;
#pragma unroll
                    for (int t = 0; t < D; ++t) {
                        const float x = h ? X[pp][t].y : X[pp][t].x;
                        r2 = fmaf(x, x, r2);
                    }
                    const float L = (h ? M[pp].y : M[pp].x) + (float)((int)(__float_as_uint(S) >> 23) - 127);
                    if (q[pp] + h < nq) V = fmaxf(V, S >= 1.17549435e-38f ? fmaf(k, r2, -L) : INFINITY);
                }
            }
            thr = -t1 - warp_max_f(V);
        }
        if (stage_end)
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
                Sd[pp].x += (double)Sf[pp].x;
                Sd[pp].y += (double)Sf[pp].y;
                Sf[pp] = make_float2(0.f, 0.f);
            }
    }
#pragma unroll
    for (int pp = 0; pp < PP; ++pp) {
        Sd[pp].x += (double)Sf[pp].x;
        Sd[pp].y += (double)Sf[pp].y;
        *reinterpret_cast<float4 *>(part + (int64_t)kc * nq_pad + q[pp]) =
            make_float4(M[pp].x, (float)Sd[pp].x, M[pp].y, (float)Sd[pp].y);
    }
}

template <int D, int TPP>
__global__ void __launch_bounds__(MS_THREADS, TPP == 2 ? 6 : 8)
    k_grad_skip(const float4 *__restrict__ tquad, const int *__restrict__ perm, const double *__restrict__ nu,
                int64_t n, const float4 *__restrict__ pquad, int64_t nq, int64_t chunk, float k, float kdiam2,
                float t2, double *__restrict__ part2, int64_t stride) {
    pdl_enter();
    __shared__ __align__(16) float4 s_p[MS_WARPS][64];   // queue: at most 31 + 32 points
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *const T = s_p[warp];
    const int64_t i0 = ((int64_t)blockIdx.x * MS_WARPS + warp) * (64 * TPP);
    if (i0 >= n) return;
    const int64_t p_begin = (int64_t)blockIdx.y * chunk, p_end = min(nq, p_begin + chunk);
    const float inv2k = 0.5f / k;
    float2 W0[TPP], W1[TPP], W2[TPP], C[TPP], acc[TPP];
    double2 acc64[TPP];
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    float V = -INFINITY, bmax = 0.f;
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) {
        const int64_t i = i0 + 64 * tp + 2 * lane;
        float4 r[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = perm[i + h];
            r[h] = tquad[j];
            if (i + h >= n) continue;
            const float x[3] = {r[h].x, r[h].y, r[h].z};
#pragma unroll
            for (int t = 0; t < D; ++t) lo[t] = fminf(lo[t], x[t]), hi[t] = fmaxf(hi[t], x[t]);
            const float B = fmaf(fmaf(x[0], x[0], fmaf(x[1], x[1], x[2] * x[2])), 0.5f * inv2k, r[h].w);
            V = fmaxf(V, B - __log2f((float)nu[j]));
            bmax = fmaxf(bmax, fabsf(B));
        }
        W0[tp] = make_float2(r[0].x, r[1].x);
        W1[tp] = make_float2(r[0].y, r[1].y);
        W2[tp] = make_float2(r[0].z, r[1].z);
        C[tp] = make_float2(r[0].w, r[1].w);
        acc[tp] = make_float2(0.f, 0.f);
        acc64[tp] = make_double2(0.0, 0.0);
    }
    const Box box = make_box<D>(lo, hi, inv2k, k);   // positions
    const float thr = -t2 - warp_max_f(V);
    const float err = warp_max_f(bmax) + kdiam2;
    const auto load = [&](int64_t g) { return g + lane < p_end ? pquad[g + lane] : make_float4(0.f, 0.f, 0.f, kPadC); };
    float4 nxt = load(p_begin);
    int have = 0;
#pragma unroll 1
    for (int64_t g = p_begin; g < p_end; g += 32) {
        const float4 p = nxt;
        nxt = load(g + 32);
        const float A = fmaf(fmaf(p.x, p.x, fmaf(p.y, p.y, p.z * p.z)), k, p.w);
        const float bound = box_bound<D>(box, p, A) + 0x1p-19f * (fabsf(A) + err);
        // a point without mass (or padding) has u = -1e30
        const bool need = p.w > 0.5f * kPadC && bound >= thr;
        const unsigned m = __ballot_sync(0xffffffffu, need);
        // the points that remain queue up in their order; a full queue of 32 is summed
        if (need) T[have + __popc(m & ((1u << lane) - 1u))] = p;
        have += __popc(m);
        __syncwarp();
        const bool flush = (g - p_begin + 32) % P2_TS == 0 || g + 32 >= p_end;
        if (have >= 32 || flush) {
            const int cnt = flush ? have : 32;
#pragma unroll 4
            for (int i = 0; i < cnt; ++i) {
                const float4 v = T[i];
                const float2 x0 = both(v.x), x1 = both(v.y), x2 = both(v.z), u = both(v.w);
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
            have -= cnt;
            __syncwarp();
            if (lane < have) T[lane] = T[32 + lane];   // at most 31 remain after a full queue
            __syncwarp();
        }
        if (flush)
#pragma unroll
            for (int tp = 0; tp < TPP; ++tp) {
                acc64[tp].x += (double)acc[tp].x;
                acc64[tp].y += (double)acc[tp].y;
                acc[tp] = make_float2(0.f, 0.f);
            }
    }
#pragma unroll
    for (int tp = 0; tp < TPP; ++tp) {
        const int64_t i = i0 + 64 * tp + 2 * lane;
        double *const o = part2 + (int64_t)blockIdx.y * stride;
        if (i < n) o[perm[i]] = acc64[tp].x;
        if (i + 1 < n) o[perm[i + 1]] = acc64[tp].y;
    }
}

// pairs of rows per thread: two where that leaves a few warps per scheduler, else one
// (four: fewer tests, but wider boxes and half the warps; 786,432 x 65,536 at eps 1e-3:
// 3.58 and 3.76 ms with four, 3.39 and 3.43 with two, 6.35 and 6.04 with one)
int rows_per_thread(int64_t rows, int64_t splits, int num_sms) {
    int pp = 2;
    while (pp > 1 && (rows + 64 * pp - 1) / (64 * pp) * splits < (int64_t)num_sms * 32) pp /= 2;
    return pp;
}

}  // namespace

void mskip_free(rsot_problem *p) {
    cudaFree(p->ms_buf);
    p->ms_buf = nullptr;
}

// Which passes leave pairs out: bit 0 pass 1, bit 1 pass 2; 0 in the solver, where the
// caller has chosen a pair kernel (RSOT_PAIRS_FP32 takes every pair) and where
// few pairs can be left out (kd = k diam^2, in 3-D a pair's reach is about
// sqrt(78 / kd) of the diameter) or the work is too small for the loops over masks and
// the first, whole stage.  Both sides in us:
//   either, 1e9 pairs: with less, a problem's first call pays for the orders (~0.3 ms)
//     what many later ones save (98,304 x 4,096: kd 4328 105 -> 95 and 84 -> 79)
//   pass 1, kd >= 700 and kd x targets per chunk >= 2e6:
//     786,432 x 65,536: kd 2164 8439 -> 3392, 721 8382 -> 7107, 433 8375 -> 9096 (not)
//     331,776 x 16,384 (2,048 per chunk): kd 2164 970 -> 568, 1082 952 -> 785, 721 946 -> 935
//     192,000 x 10,000 (1,024): kd 2164 364 -> 267;  61,206 x 5,003 (512): kd 2885 61 -> 73 (not)
//   pass 2, kd >= 500:
//     786,432 x 65,536: kd 2164 8458 -> 3428, 721 8456 -> 6669, 433 8457 -> 8452 (not)
//     192,000 x 10,000: kd 1082 373 -> 346;  60,000 x 20,000: kd 2885 188 -> 92
//     61,206 x 5,003: kd 2885 51.1 -> 51.2 (not)
static int mskip_passes(const rsot_problem *p, double eps) {
    const double kappa = kLog2e / (2.0 * eps), kd = kappa * p->diam2;
    if (p->in_solve || p->pair_kernel != 2 || !(kd <= 0x1p20) || !skip_estimate_fits(p, kappa)) return 0;
    if ((double)p->nq * (double)p->n < 1e9) return 0;
    return (kd >= 700.0 && kd * (double)p->chunk1 >= 2e6 ? 1 : 0) | (kd >= 500.0 ? 2 : 0);
}

static bool mskip_alloc(rsot_problem *p) {
    if (p->ms_buf) return true;
    const int64_t blk = 128 * MS_WARPS, tiles = p->nq_pad / P2_TS, units = (p->n + blk - 1) / blk;
    // pass 2 in about 60 CTAs per SM where that many stages exist: skipping leaves
    // their work uneven; at most 64 splits (the last kernel's sums)
    const int64_t want = std::min({tiles, (60 * p->num_sms + units - 1) / units, (int64_t)64});
    p->ms_chunk2 = (tiles + want - 1) / want * P2_TS;
    p->ms_s2 = (int)((p->nq_pad + p->ms_chunk2 - 1) / p->ms_chunk2);
    // rows are read in whole warps of 64 or 128: the orders are padded to that (1,024s)
    const size_t np = (size_t)p->nq_pad, nt = (size_t)p->n_pad;
    // the orders, then pass 2's partials, whose place is scratch while the orders are made
    const size_t part = std::max({nt * 8 * p->ms_s2, cell_order_scratch(p->n), cell_order_scratch((p->nq + 1) / 2)});
    char *b = nullptr;
    if (cudaMalloc(&b, np / 2 * 4 + nt * 4 + part) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    p->ms_buf = b;
    p->ms_perm_q = reinterpret_cast<int *>(b);
    p->ms_perm_t = p->ms_perm_q + np / 2;
    p->ms_part2 = reinterpret_cast<double *>(p->ms_perm_t + nt);
    // points by pairs, which share a raise of their shifts
    cudaError_t e = cell_order(p, p->x64, (p->nq + 1) / 2, p->nq_pad / 2, p->ms_perm_q, p->ms_part2, 2);
    if (!e) e = cell_order(p, p->y64, p->n, p->n_pad, p->ms_perm_t, p->ms_part2);
    // once per problem: a later evaluation may run on another stream
    if (!e) e = cudaStreamSynchronize(p->stream);
    if (e) {
        cudaGetLastError();
        mskip_free(p);
        return false;
    }
    return true;
}

// that choice with its buffers and orders, which are made once per problem; without
// memory for them the dense passes run
int mskip_ready(rsot_problem *p, double eps) {
    const int passes = mskip_passes(p, eps);
    return passes && mskip_alloc(p) ? passes : 0;
}

template <int D>
static void mskip_lse_d(rsot_problem *p, double eps) {
    const float k = (float)(kLog2e / (2.0 * eps)), kd = (float)(kLog2e / (2.0 * eps) * p->diam2);
    const int pp = rows_per_thread(p->nq, p->k1, p->num_sms);
    dim3 g((unsigned)((p->nq + 64 * pp * MS_WARPS - 1) / (64 * pp * MS_WARPS)), (unsigned)p->k1);
    auto f = pp == 2 ? k_lse_skip<D, 2> : k_lse_skip<D, 1>;
    launch_pdl(false, f, g, MS_THREADS, 0, p->stream, p->xs, p->ms_perm_q, p->nq, p->nq_pad,
               p->tquad, (int)p->n, p->chunk1, k, kd, (float)(61.0 + log2((double)p->n)), p->part1);
}
void mskip_lse(rsot_problem *p, double eps) { (p->d == 3 ? mskip_lse_d<3> : mskip_lse_d<2>)(p, eps); }

template <int D>
static void mskip_grad_d(rsot_problem *p, double eps) {
    const float k = (float)(kLog2e / (2.0 * eps)), kd = (float)(kLog2e / (2.0 * eps) * p->diam2);
    const int pp = rows_per_thread(p->n, p->ms_s2, p->num_sms);
    dim3 g((unsigned)((p->n + 64 * pp * MS_WARPS - 1) / (64 * pp * MS_WARPS)), (unsigned)p->ms_s2);
    auto f = pp == 2 ? k_grad_skip<D, 2> : k_grad_skip<D, 1>;
    launch_pdl(false, f, g, MS_THREADS, 0, p->stream, p->tquad, p->ms_perm_t, p->nu, p->n,
               p->pquad, p->nq, p->ms_chunk2, k, kd, (float)(61.0 + log2((double)p->nq)), p->ms_part2, p->n_pad);
}
void mskip_grad(rsot_problem *p, double eps) { (p->d == 3 ? mskip_grad_d<3> : mskip_grad_d<2>)(p, eps); }

}  // namespace rsot
