// Compensated dense evaluation returned to a caller (RSOT_COMPENSATED outside
// rsot_solve).
//
// The same quantities as the passes of rsot_df.cu -- exponents as double-float
// sums in the log2 domain, r_qj = c_j + x'_q.w_j, ex2.approx of the head with
// a first-order tail, Kahan sums within a tile, FP64 across -- with the same
// error budget (RSOT_COMPENSATED_GRAD_REL), in two thirds of the operations
// and for the pairs that matter only:
//   * Operands are split on grids so that the leading sums need no error terms.
//     With |x'| <= P = 2^p, |w| <= Q = 2^q: x = x1 + x2 + x3, x1 a multiple of
//     2^(p-10), x2 of 2^(p-22), x3 the rest in FP32, xh = x1 + x2; w and c
//     alike (c1 a multiple of 2^(p+q-20), c2 of 2^(p+q-32)).
//       s1 = c1 + sum x1 w1             exact while |c| <= 13 P Q
//       s2 = c2 + sum x1 w2 + x2 w1     exact (below 2^(p+q-8))
//       s3 = c3 + sum xh w3 + x3 wh + x2 w2   rounded, error < 2^(p+q-41)
//     fl(s1 + s2), its exact error plus s3, and one renormalisation give r's head
//     and tail: 6 d + 7 operations instead of 12 d + 3 (products and their errors
//     summed by TwoSum).  The head is the one that rsot_df.cu forms but for a few
//     ties, so ex2.approx sees the same arguments and the results agree to 1e-10
//     (head = fl(s1 + fl(s2 + s3)), two operations less, missed more ties: 7e-10).
//   * The shift M of pass 1 is integral, so that head - M needs three operations
//     for its error term instead of six.  It is the running ceiling of the
//     maximum as in rsot_df.cu (a column chunk starts from the FP32 maximum over
//     the columns before it, rsot_skip.cu): with the final maximum instead, the
//     rounding of head - M, and with it ex2.approx's argument, differed for the
//     first columns of a row (gradients then differ by up to 1e-9, their error
//     being 2e-9).
//   * Columns all of whose pairs with a warp's 64 rows cannot change a sum by
//     2^-60 of it are skipped (rsot_skip.cuh).
// Where an operand leaves the ranges above the records kernel raises
// kErrRange64 and the caller runs the passes of rsot_df.cu; rsot_solve always
// does, so that its iterates keep their bits.
#include <math.h>

#include <algorithm>

#include "rsot_internal.cuh"
#include "rsot_inner.cuh"
#include "rsot_skip.cuh"

namespace rsot {

namespace {

constexpr int CX_THREADS = 128;
constexpr int CX_ROWS = 2 * CX_THREADS;
constexpr int CX_TS = 128;       // columns per shared-memory tile
constexpr float kExcl = -1.0e30f;

typedef float2 f2;
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }
// a - b rounded once: the product b * -1 is exact
__device__ __forceinline__ f2 sub2(f2 a, f2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// (v1, v2, v3, v1 + v2) of the three coordinates, and (c1, c2, c3, 0) of a
// target or (u head, u tail, 0, 0) of a point
struct __align__(16) CxRec {
    float4 v[3];
    float4 s;
};

// v on the grids g1, g2 (powers of two)
__device__ __forceinline__ float4 split3(double v, double g1, double g2) {
    const double a = rint(v / g1) * g1, b = rint((v - a) / g2) * g2;
    return make_float4((float)a, (float)b, (float)((v - a) - b), (float)(a + b));
}

__global__ void k_cx_points(const double *__restrict__ x64, int64_t nq, int64_t nq_pad, int d, double P,
                            CxRec *__restrict__ prec) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nq_pad) return;
    CxRec r;
    for (int t = 0; t < 3; ++t)
        r.v[t] = i < nq && t < d ? split3(x64[i * d + t], P * 0x1p-10, P * 0x1p-22)
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
    r.s = make_float4(kExcl, 0.f, 0.f, 0.f);
    prec[i] = r;
}

// targets: w_j = 2k y'_j, c_j = b_j - k |y'_j|^2 as rsot_df.cu forms them
__global__ void k_cx_targets(const double *__restrict__ psi, const double *__restrict__ y64,
                             const double *__restrict__ lnu, int64_t n, int64_t n_pad, int d, double eps,
                             double P, double Q, double kappa_diam2, CxRec *__restrict__ trec,
                             EvalResult *__restrict__ res) {
    pdl_enter();
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_pad) return;
    const double k = kLog2e / (2.0 * eps);
    CxRec r;
    for (int t = 0; t < 3; ++t) r.v[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    r.s = make_float4(kExcl, 0.f, 0.f, 0.f);
    if (j < n) {
        const double b = ((psi[j] - psi[0]) / eps + lnu[j]) * kLog2e;
        double yy = 0.0;
        for (int t = 0; t < d; ++t) {
            const double yt = y64[j * d + t];
            r.v[t] = split3(2.0 * k * yt, Q * 0x1p-10, Q * 0x1p-22);
            yy += yt * yt;
        }
        const double c = b - k * yy;
        r.s = split3(c, P * Q * 0x1p-20, P * Q * 0x1p-32);
        // 7 roundings of 2^-24 of the terms' magnitudes bound the FP32 estimate
        const double E = 0x1p-20 * (fabs(b) + kappa_diam2);
        if (!(fabs(c) <= 13.0 * P * Q) || !(E <= 16.0)) atomicOr(&res->flags, kErrRange64);
    }
    trec[j] = r;
}

struct CxOp {   // the thread's two rows
    f2 v1[3], v2[3], v3[3], vh[3];
};

// head and tail of r for one column and the two rows
template <int D>
__device__ __forceinline__ void cx_exponent(const CxOp &R, const CxRec &B, f2 s1, f2 s2, f2 s3, f2 &rh,
                                            f2 &rt) {
#pragma unroll
    for (int t = 0; t < D; ++t) {
        const float4 b = B.v[t];
        s1 = fma2(R.v1[t], both(b.x), s1);
        s2 = fma2(R.v1[t], both(b.y), s2);
        s2 = fma2(R.v2[t], both(b.x), s2);
        s3 = fma2(R.vh[t], both(b.z), s3);
        s3 = fma2(R.v3[t], both(b.w), s3);
        s3 = fma2(R.v2[t], both(b.y), s3);
    }
    const f2 h = add2(s1, s2);
    const f2 lo = add2(sub2(s2, sub2(h, s1)), s3);   // its error exactly, plus s3: below one ulp or two
    rh = add2(h, lo);
    rt = sub2(lo, sub2(rh, h));
}

__device__ __forceinline__ void cx_load(const CxRec &a, const CxRec &b, CxOp &R) {
    for (int t = 0; t < 3; ++t) {
        R.v1[t] = make_float2(a.v[t].x, b.v[t].x);
        R.v2[t] = make_float2(a.v[t].y, b.v[t].y);
        R.v3[t] = make_float2(a.v[t].z, b.v[t].z);
        R.vh[t] = make_float2(a.v[t].w, b.v[t].w);
    }
}

// s += e (Kahan), cs += e w
__device__ __forceinline__ void cx_sum(f2 &s, f2 &comp, f2 &cs, f2 e, f2 w) {
    const f2 y = sub2(e, comp);
    const f2 t = add2(s, y);
    comp = sub2(sub2(t, s), y);
    s = t;
    cs = fma2(e, w, cs);
}

// one column: the exponents of the thread's two rows, their exponentials and sums
template <int D, int PASS>
__device__ __forceinline__ void cx_column(const CxOp &W, const CxRec &B, f2 C1, f2 C2, f2 C3, f2 &M,
                                          f2 &s, f2 &comp, f2 &cs, double &acc0, double &acc1) {
    f2 rh, rt;
    if (PASS == 1) {
        cx_exponent<D>(W, B, both(B.s.x), both(B.s.y), both(B.s.z), rh, rt);
        if (rh.x > M.x || rh.y > M.y) {   // raise a shift to ceil(r): exact rescaling
            const float mx = rh.x > M.x ? ceilf(rh.x) : M.x, my = rh.y > M.y ? ceilf(rh.y) : M.y;
            const f2 f = make_float2(pow2_int_f(M.x - mx), pow2_int_f(M.y - my));
            acc0 *= pow2_int_d(M.x - mx);
            acc1 *= pow2_int_d(M.y - my);
            s = __fmul2_rn(s, f);
            comp = __fmul2_rn(comp, f);
            cs = __fmul2_rn(cs, f);
            M = make_float2(mx, my);
        }
        // M is integral: rh - (a + M) is the rounding error of a exactly
        const f2 a = sub2(rh, M);
        const f2 w = add2(sub2(rh, add2(a, M)), rt);
        cx_sum(s, comp, cs, make_float2(ex2_approx(a.x), ex2_approx(a.y)), w);
    } else {
        cx_exponent<D>(W, B, C1, C2, C3, rh, rt);
        const f2 uh = both(B.s.x);
        const f2 a = add2(rh, uh);   // TwoSum
        const f2 bb = sub2(a, rh);
        const f2 w = add2(sub2(rh, sub2(a, bb)), sub2(uh, bb));
        cx_sum(s, comp, cs, make_float2(ex2_approx(a.x), ex2_approx(a.y)), add2(add2(w, rt), both(B.s.y)));
    }
}

// rows and columns of a pass: split records, FP32 records, values of the ball
// test (rsot_skip.cuh) and the factors that turn the FP32 records into positions
struct CxRows {
    const CxRec *rec;
    const float4 *f;
    const float *val;
    const int *perm;    // row order (null: as stored)
    float slack, scale;
    int64_t count, pad;
};
struct CxCols {
    const CxRec *rec;
    const float4 *f;
    const float *val;
    float scale;
    int64_t count;
};

// PASS 1: rows = points (two consecutive ones per thread), columns = targets,
// out[chunk][row] = sum 2^(r - M), M in shift; PASS 2: rows = targets (in the order of
// perm), columns = points, out = sum 2^(r + u) = sum m_q p_qj.  Bound by
// register reads: 6 d + 16 (pass 1) or 6 d + 20 packed operations per two pairs,
// 48 and 52 cycles a pair and warp at d = 3 where all pairs count (70 and 59 in
// rsot_df.cu).
template <int D, int PASS>
__global__ void __launch_bounds__(CX_THREADS)
    k_cx_pass(CxRows rows, CxCols cols, int64_t chunk, const float *__restrict__ pmax, float kappa,
              float kdiam2, double *__restrict__ out, float *__restrict__ shift,
              const EvalResult *__restrict__ res) {
    pdl_enter();
    if (res->flags & kErrRange64) return;
    __shared__ CxRec s_rec[CX_TS];
    __shared__ __align__(16) float4 s_f[CX_TS];
    __shared__ float s_v[CX_TS];
    const int tid = threadIdx.x, lane = tid & 31;
    const float margin = 2.0f * skip_error(res, kdiam2);
    const int64_t i0 = (int64_t)blockIdx.x * CX_ROWS + 2 * tid;   // < rows.pad, a multiple of 1,024
    // pass 1: order of point pairs, pass 2: of targets (null: as stored); points in cell
    // order, pass 1 of 98,304 x 65,536 at eps 1e-3: 1.95 -> 1.77 ms
    int64_t at0 = i0, at1 = i0 + 1;
    if (rows.perm) {
        at0 = PASS == 1 ? 2 * rows.perm[i0 >> 1] : rows.perm[i0];
        at1 = PASS == 1 ? at0 + 1 : rows.perm[i0 + 1];
    }
    const bool in0 = (PASS == 1 ? at0 : i0) < rows.count, in1 = (PASS == 1 ? at1 : i0 + 1) < rows.count;
    CxOp W;
    f2 C1, C2, C3, X[3], thr, M;
    RowBall ball;
    {
        const CxRec a = rows.rec[at0], b = rows.rec[at1];
        cx_load(a, b, W);
        C1 = make_float2(a.s.x, b.s.x);
        C2 = make_float2(a.s.y, b.s.y);
        C3 = make_float2(a.s.z, b.s.z);
        const float4 fa = rows.f[at0], fb = rows.f[at1];
        X[0] = make_float2(fa.x, fb.x);
        X[1] = make_float2(fa.y, fb.y);
        X[2] = make_float2(fa.z, fb.z);
        const float va = in0 ? rows.val[at0] + rows.slack + margin : -INFINITY;
        const float vb = in1 ? rows.val[at1] + rows.slack + margin : -INFINITY;
        ball = row_ball(fa, va, fb, vb, rows.scale);
        thr = make_float2(fa.w - margin, fb.w - margin);   // +inf: padding
        M = make_float2(-INFINITY, -INFINITY);
        if (PASS == 1)
            for (int k = 0; k < (int)blockIdx.y; ++k) {
                const float2 m = *reinterpret_cast<const float2 *>(pmax + (int64_t)k * rows.pad + at0);
                M = make_float2(fmaxf(M.x, ceilf(m.x)), fmaxf(M.y, ceilf(m.y)));
            }
    }
    const int64_t c_begin = (int64_t)blockIdx.y * chunk;
    const int64_t c_end = min(cols.count, c_begin + chunk);
    double acc0 = 0.0, acc1 = 0.0;
    for (int64_t t0 = c_begin; t0 < c_end; t0 += CX_TS) {
        const int cnt = (int)min((int64_t)CX_TS, c_end - t0);
        __syncthreads();
        if (tid < cnt) {
            s_f[tid] = cols.f[t0 + tid];
            s_v[tid] = cols.val[t0 + tid];
        }
        for (int i = tid; i < cnt * 4; i += CX_THREADS)
            reinterpret_cast<float4 *>(s_rec)[i] = reinterpret_cast<const float4 *>(cols.rec + t0)[i];
        __syncthreads();
        f2 s = make_float2(0.f, 0.f), comp = s, cs = s;
        bool any = false;
        for (int g = 0; g < cnt; g += 32) {
            unsigned need = __ballot_sync(
                0xffffffffu,
                g + lane < cnt && ball_needs(ball, s_f[g + lane], s_v[g + lane], cols.scale, kappa));
            // most pairs of a group that the ball keeps whole are needed: no pair test
            if (need == 0xffffffffu) {
                any = true;
#pragma unroll 2
                for (int c = g; c < g + 32; ++c)
                    cx_column<D, PASS>(W, s_rec[c], C1, C2, C3, M, s, comp, cs, acc0, acc1);
                continue;
            }
            for (; need; need &= need - 1) {
                const int c = g + __ffs(need) - 1;
                const f2 est = pair_exponent<D>(X, s_f[c]);
                if (!__any_sync(0xffffffffu, est.x >= thr.x || est.y >= thr.y)) continue;
                any = true;
                cx_column<D, PASS>(W, s_rec[c], C1, C2, C3, M, s, comp, cs, acc0, acc1);
            }
        }
        if (any) {
            acc0 += ((double)s.x - (double)comp.x) + kLn2 * (double)cs.x;
            acc1 += ((double)s.y - (double)comp.y) + kLn2 * (double)cs.y;
        }
    }
    out[(int64_t)blockIdx.y * rows.pad + at0] = acc0;
    out[(int64_t)blockIdx.y * rows.pad + at1] = acc1;
    if (PASS == 1) *reinterpret_cast<float2 *>(shift + (int64_t)blockIdx.y * rows.pad + at0) = M;
}

// R_q, the J term of the point's mass, and the column of pass 2: u_q = log2 m_q
// - R_q, (x', -R_q) and A_q
__global__ void k_cx_combine(const double *__restrict__ part, const float *__restrict__ shift, int k1,
                             int64_t nq, int64_t nq_pad, float t1,
                             const double *__restrict__ lmass2, const double *__restrict__ mass,
                             const float4 *__restrict__ ptrow, CxRec *__restrict__ prec,
                             float4 *__restrict__ ptcol, float *__restrict__ ptA,
                             double *__restrict__ lse_buf, double *__restrict__ blockJ) {
    pdl_enter();
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double contrib = 0.0;
    if (q < nq) {
        double S = 0.0;
        float M = -INFINITY;   // the last chunk's is the largest
        for (int k = 0; k < k1; ++k) M = fmaxf(M, shift[(int64_t)k * nq_pad + q]);
        for (int k = 0; k < k1; ++k) {
            const double v = part[(int64_t)k * nq_pad + q];
            if (v > 0.0) S += v * pow2_int_d(shift[(int64_t)k * nq_pad + q] - M);
        }
        const float4 x = ptrow[q];
        const double R = (double)M + log2(S);
        lse_buf[q] = R;
        float4 col = make_float4(x.x, x.y, x.z, kPadC);
        float A = -INFINITY;
        if (mass[q] > 0.0) {
            contrib = mass[q] * R;
            const double u = lmass2[q] - R;
            const float uh = (float)u;
            prec[q].s.x = uh;
            prec[q].s.y = (float)(u - (double)uh);
            col.w = (float)-R;
            A = ptA[q] + (x.w + t1 - (float)R);
        }
        ptcol[q] = col;
        ptA[q] = A;
    }
    store_partial(contrib, blockJ);
}

}  // namespace

void cx_free(rsot_problem *p) {
    cudaFree(p->cx_buf);
    p->cx_buf = nullptr;
}

static bool cx_alloc(rsot_problem *p, double P) {
    if (p->cx_buf) return true;
    auto chunked = [&](int64_t rows, int64_t cols, int &split, int64_t &chunk) {
        const int64_t tiles = (cols + CX_TS - 1) / CX_TS;
        // 40 CTAs per SM: skipped columns leave their work uneven (98,304 x 65,536:
        // pass 2 2.44 ms with 5 per SM, 2.34 with 20, 2.31 with 40)
        const int64_t units = (rows + CX_ROWS - 1) / CX_ROWS;
        const int64_t want = std::min({tiles, (40 * p->num_sms + units - 1) / units, (int64_t)256});
        chunk = (tiles + want - 1) / want * CX_TS;
        split = (int)((cols + chunk - 1) / chunk);
    };
    chunked(p->n, p->nq, p->cx_s2, p->cx_chunk2);
    const size_t np = (size_t)p->nq_pad, nt = (size_t)p->n_pad;
    char *b = nullptr;
    if (cudaMalloc(&b, (np + nt) * sizeof(CxRec) + np * p->sk_k * 12 + nt * p->cx_s2 * 8) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    p->cx_buf = b;
    p->cx_prec = b;
    p->cx_trec = b + np * sizeof(CxRec);
    p->cx_part1 = reinterpret_cast<double *>(b + (np + nt) * sizeof(CxRec));
    p->cx_part2 = p->cx_part1 + np * p->sk_k;
    p->cx_shift = reinterpret_cast<float *>(p->cx_part2 + nt * p->cx_s2);
    k_cx_points<<<(unsigned)(np / 256), 256, 0, p->stream>>>(p->x64, p->nq, p->nq_pad, p->d, P,
                                                            reinterpret_cast<CxRec *>(p->cx_prec));
    // once per problem: a later evaluation may run on another stream
    if (cudaStreamSynchronize(p->stream) != cudaSuccess) {
        cudaGetLastError();
        cx_free(p);
        return false;
    }
    return true;
}

static double pow2_above(double v) {   // the power of two in (v, 2 v]
    int e = 0;
    frexp(v, &e);
    return ldexp(1.0, e);
}

bool cx_ready(rsot_problem *p, double eps) {
    if (p->in_solve || !(p->half_ext > 0.0)) return false;
    // smaller problems are bound by the launches, three more than rsot_df.cu's, against
    // its chains over the targets (us there and here: 16 x 500 71 and 78, 1,000 x 500 76 and
    // 90, 12,000 x 300 84 and 94; 16 x 1,000 97 and 79, 1,000 x 1,000 104 and 93, 12,000 x
    // 1,000 121 and 111, 3,000 x 1,500 164 and 104, 16 x 65,536 3,713 and 169; from 2.5e7
    // pairs 200,000 x 128 487 and 231)
    if (p->n < 1000 && (double)p->nq * (double)p->n < 2.5e7) return false;
    const double P = pow2_above(p->half_ext), Q = pow2_above(kLog2e / eps * p->half_ext);
    // all grids and sums inside FP32's range; the estimate's error bound below 16
    if (!(P >= 0x1p-40 && P <= 0x1p40 && P * Q >= 0x1p-40 && P * Q <= 0x1p40)) return false;
    return skip_ready(p, eps) && cx_alloc(p, P);
}

template <int D>
static void cx_passes(rsot_problem *p, double eps, float t1, float kd) {
    cudaStream_t st = p->stream;
    CxRec *prec = reinterpret_cast<CxRec *>(p->cx_prec), *trec = reinterpret_cast<CxRec *>(p->cx_trec);
    const double k = kLog2e / (2.0 * eps);
    const float kappa = (float)k, inv2k = (float)(0.5 / k);
    const float tmax = (float)(60.0 + log2(p->msum / p->nu_min));   // largest slack of a target
    trace_begin(p, "lse_cx");
    const CxRows pr = {prec, p->sk_ptrow, p->sk_ptA, p->sk_perm_q, t1, 1.f, p->nq, p->nq_pad};
    const CxCols tc = {trec, p->tquad, p->sk_tgB, inv2k, p->n};
    // the column chunks of the maximum's kernel: a chunk's shift starts from theirs
    k_cx_pass<D, 1><<<dim3((unsigned)((p->nq + CX_ROWS - 1) / CX_ROWS), (unsigned)p->sk_k), CX_THREADS, 0,
                      st>>>(pr, tc, p->sk_chunk, p->sk_part, kappa, kd, p->cx_part1, p->cx_shift,
                            p->res_dev);
    trace_end(p);
    trace_begin(p, "combine_cx");
    const unsigned th = p->per_comb == 1 ? 256 : kSmall;
    launch_pdl(true, k_cx_combine, (unsigned)(p->nq_pad / th), th, 0, st, p->cx_part1, p->cx_shift, p->sk_k, p->nq,
                                                              p->nq_pad, t1, p->lmass2, p->mass, p->sk_ptrow, prec,
                                                              p->sk_ptcol, p->sk_ptA, p->lse_buf, p->blockJ);
    trace_end(p);
    trace_begin(p, "grad_cx");
    const CxRows tr = {trec, p->sk_tgrow, p->sk_tgB, p->sk_perm, tmax, inv2k, p->n, p->n_pad};
    const CxCols pc = {prec, p->sk_ptcol, p->sk_ptA, 1.f, p->nq};
    k_cx_pass<D, 2><<<dim3((unsigned)((p->n + CX_ROWS - 1) / CX_ROWS), (unsigned)p->cx_s2), CX_THREADS, 0,
                      st>>>(tr, pc, p->cx_chunk2, nullptr, kappa, kd, p->cx_part2, nullptr, p->res_dev);
    trace_end(p);
}

cudaError_t launch_compensated_cx(rsot_problem *p, const double *psi, double eps, double *grad) {
    cudaStream_t st = p->stream;
    const double P = pow2_above(p->half_ext), Q = pow2_above(kLog2e / eps * p->half_ext);
    const double kd = kLog2e / (2.0 * eps) * p->diam2;
    cudaError_t e = launch_skip(p, psi, eps);
    if (e) return e;
    trace_begin(p, "prep_cx");
    const unsigned tt = small_threads(p->n_pad, p->num_sms);
    launch_pdl(true, k_cx_targets, (unsigned)(p->n_pad / tt), tt, 0, st, psi, p->y64, p->lnu, p->n, p->n_pad, p->d,
                                                            eps, P, Q, kd,
                                                            reinterpret_cast<CxRec *>(p->cx_trec),
                                                            p->res_dev);
    trace_end(p);
    (p->d == 3 ? cx_passes<3> : cx_passes<2>)(p, eps, (float)skip_t1(p), (float)kd);
    if ((e = cudaGetLastError())) return e;
    return launch_finalize(p, psi, eps,
                           {p->cx_part2, p->cx_s2, p->n_pad, nullptr, p->blockJ, (int)(p->nq_pad / 256), p->per_comb, 1,
                            p->per_prep},
                           grad);
}

}  // namespace rsot
