// Transport maps (Sec. 6.3), conditional centroids (Eq. barycenter_fixed_point)
// and the damped Lloyd iteration for barycenters (Eq. damped_lloyd, Sec. 6.2).
//
// Both maps and centroids are sums over the plan p_qj of Eq. final_plan_density,
// evaluated like the mixed dense passes (rsot_dense.cu: log2 domain, translated
// coordinates, r_qj = c_j + x'_q.w_j with w_j = 2k y'_j, FP32 pair arithmetic,
// FP64 across tiles):
//   T_bary(x_q) - o = sum_j 2^(r_qj - M) w_j / (2k sum_j 2^(r_qj - M))   (per point,
//                     an online max shift M as in pass 1)
//   j*(q)           = argmax_j r_qj  (the first maximum in index order)
//   a_j             = sum_q m_q p_qj = sum_q 2^(r_qj + u_q),  u_q = log2 m_q - R_q
//   T_j             = (sum_q m_q p_qj x'_q + o a_j) / nu_j               (per target,
//                     after a dense evaluation provides u_q)
// The centroids' sums are formed by pass 2 of the evaluation, whose exponents they
// share (rsot_dense.cu, k_grad_mixed); the maps take a pass of their own over the
// target records on the CUDA cores.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <chrono>
#include <vector>

#include "rsot_internal.cuh"
#include "rsot_inner.cuh"

namespace rsot {
namespace {

constexpr int MP_THREADS = 64;    // maps: two points per thread
constexpr int MP_TS = 256;        // target records per shared-memory tile
constexpr int MP_SUB = 16;        // targets per max sub-tile
constexpr int CT_TARGETS = 64;    // centroids: targets per block of the last kernel

struct Origin {
    double o[3];
};

inline int64_t round_up(int64_t a, int64_t b) { return (a + b - 1) / b * b; }

// T_bary and j* per point over all target records (of the dense pass 1:
// (w0,w1,w2,c)); n_rec is a multiple of MP_TS.  A thread holds two neighbouring
// points, whose arithmetic is packed (bound: the packed instructions' register
// reads, about 25 cycles per sub-partition for 32 x 2 pairs), and looks for the
// maximum's index only in a sub-tile whose maximum exceeds the one before: 98,304
// x 4,096 took 274 us with one point per thread and a select per pair, 166 now.
template <int D>
__global__ void __launch_bounds__(MP_THREADS)
    k_maps(const float *__restrict__ xs, int64_t nq_pad, int64_t nq, const float4 *__restrict__ tquad,
           int64_t n_rec, int64_t n, double inv2k, Origin origin, const EvalResult *__restrict__ res,
           double *__restrict__ Tout, int64_t *__restrict__ jout) {
    __shared__ __align__(16) float4 sm[MP_TS];
    const int64_t q = 2 * ((int64_t)blockIdx.x * MP_THREADS + threadIdx.x);   // nq_pad is even
    float2 X[3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
        X[k] = k < D && q < nq_pad ? *reinterpret_cast<const float2 *>(xs + k * nq_pad + q) : make_float2(0.f, 0.f);
    float M[2] = {-INFINITY, -INFINITY}, best[2] = {-INFINITY, -INFINITY};
    int64_t bj[2] = {0, 0};
    double S[2] = {0.0, 0.0}, A[D][2];
#pragma unroll
    for (int k = 0; k < D; ++k) A[k][0] = A[k][1] = 0.0;
    for (int64_t t0 = 0; t0 < n_rec; t0 += MP_TS) {
        __syncthreads();
        for (int i = threadIdx.x; i < MP_TS; i += MP_THREADS) sm[i] = tquad[t0 + i];
        __syncthreads();
        float2 s = make_float2(0.f, 0.f), a[D];
#pragma unroll
        for (int k = 0; k < D; ++k) a[k] = s;
#pragma unroll 1
        for (int u0 = 0; u0 < MP_TS; u0 += MP_SUB) {
            float2 r[MP_SUB];
            float mx[2] = {-INFINITY, -INFINITY};
#pragma unroll
            for (int i = 0; i < MP_SUB; ++i) {
                r[i] = pair_exponent<D>(X, sm[u0 + i]);
                mx[0] = fmaxf(mx[0], r[i].x);
                mx[1] = fmaxf(mx[1], r[i].y);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (!(mx[h] > best[h])) continue;   // strict: the first maximum in index order
                best[h] = mx[h];
                int at = 0;
#pragma unroll
                for (int i = MP_SUB - 1; i >= 0; --i)
                    if ((h ? r[i].y : r[i].x) == mx[h]) at = i;
                bj[h] = t0 + u0 + at;
                if (mx[h] > M[h]) {   // raise the shift to ceil(max), rescale by a power of two
                    const float mn = ceilf(mx[h]);
                    if (M[h] != -INFINITY) {
                        const float dl = M[h] - mn, f = pow2_int_f(dl);
                        const double dd = pow2_int_d(dl);
                        (h ? s.y : s.x) *= f;
                        S[h] *= dd;
#pragma unroll
                        for (int k = 0; k < D; ++k) {
                            (h ? a[k].y : a[k].x) *= f;
                            A[k][h] *= dd;
                        }
                    }
                    M[h] = mn;
                }
            }
            const float2 nm = make_float2(-M[0], -M[1]);
#pragma unroll
            for (int i = 0; i < MP_SUB; ++i) {
                const float4 w = sm[u0 + i];
                const float2 t = __fadd2_rn(r[i], nm), e = make_float2(ex2_approx(t.x), ex2_approx(t.y));
                s = __fadd2_rn(s, e);
                a[0] = __ffma2_rn(e, both(w.x), a[0]);
                a[1] = __ffma2_rn(e, both(w.y), a[1]);
                if (D == 3) a[D - 1] = __ffma2_rn(e, both(w.z), a[D - 1]);
            }
        }
        S[0] += s.x, S[1] += s.y;
#pragma unroll
        for (int k = 0; k < D; ++k) A[k][0] += a[k].x, A[k][1] += a[k].y;
    }
    if (!res->ok) return;   // outputs are written on success
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (q + h >= nq) break;
        if (jout) jout[q + h] = bj[h] < n ? bj[h] : n - 1;
        if (Tout)
#pragma unroll
            for (int k = 0; k < D; ++k) Tout[(q + h) * D + k] = origin.o[k] + A[k][h] / S[h] * inv2k;
    }
}

// T_j = (sum m p x' + o a_j) / nu_j and a_j from pass 2's partials (rows 1 .. d + 1
// of a split), one thread per target and sum, eight loads in flight, added in the
// splits' order
__global__ void __launch_bounds__(4 * CT_TARGETS)
    k_centroid_final(const double *__restrict__ part, int splits, int64_t n_pad, int64_t n, int d,
                     const double *__restrict__ nu, Origin origin, const EvalResult *__restrict__ res,
                     double *__restrict__ T, double *__restrict__ mass) {
    __shared__ double sh[4][CT_TARGETS];
    const int t = threadIdx.x % CT_TARGETS, k = threadIdx.x / CT_TARGETS;   // sum k of target t
    const int64_t j = (int64_t)blockIdx.x * CT_TARGETS + t;
    double s = 0.0;
    if (j < n && k <= d) {
        const double *p = part + (k + 1) * n_pad + j;
        const int64_t stride = (d + 2) * n_pad;
        int i = 0;
        for (; i + 8 <= splits; i += 8) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = p[(i + u) * stride];
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        for (; i < splits; ++i) s += p[i * stride];
    }
    sh[k][t] = s;
    __syncthreads();
    if (j >= n || !res->ok) return;
    if (k < d) T[j * d + k] = (s + origin.o[k] * sh[d][t]) / nu[j];
    if (k == d && mass) mass[j] = s;
}

}  // namespace

static Origin origin_of(const rsot_problem *p) { return {{p->origin[0], p->origin[1], p->origin[2]}}; }

// T_bary / j* over the dense target records of the last mixed evaluation
cudaError_t launch_maps(rsot_problem *p, double eps, double *T_dev, int64_t *j_dev) {
    const int64_t n_rec = round_up(p->n, MP_TS);
    const double inv2k = 1.0 / (2.0 * kLog2e / (2.0 * eps));
    auto f = p->d == 3 ? k_maps<3> : k_maps<2>;
    f<<<(unsigned)((p->nq + 2 * MP_THREADS - 1) / (2 * MP_THREADS)), MP_THREADS, 0, p->stream>>>(
        p->xs, p->nq_pad, p->nq, p->tquad, n_rec, p->n, inv2k, origin_of(p), p->res_dev, T_dev, j_dev);
    return cudaGetLastError();
}

// centroids from the partials of the last mixed evaluation (cent_now)
cudaError_t launch_centroids(rsot_problem *p, double *T_dev, double *mass_dev) {
    k_centroid_final<<<(unsigned)((p->n + CT_TARGETS - 1) / CT_TARGETS), 4 * CT_TARGETS, 0, p->stream>>>(
        p->cent_part, p->cent_s2, p->n_pad, p->n, p->d, p->nu, origin_of(p), p->res_dev, T_dev, mass_dev);
    return cudaGetLastError();
}

}  // namespace rsot
