// Operands of the pair skipping (rsot_skip.cuh): the largest FP32 exponent of
// every point, the records and thresholds of the tests, and the order of the
// target rows.
#include <math.h>

#include <algorithm>

#include "rsot_internal.cuh"
#include "rsot_inner.cuh"
#include "rsot_skip.cuh"

namespace rsot {
namespace {

constexpr int RM_THREADS = 128;
constexpr int RM_TS = 256;   // targets per shared-memory tile
constexpr int SORT_CELLS = 4096, SORT_THREADS = 256;

// max_j r_qj over a chunk of targets, two points per lane pair and PP pairs a
// thread (4 share a target's load; 1 where that leaves SMs idle)
template <int D, int PP>
__global__ void __launch_bounds__(RM_THREADS)
    k_row_max(const float *__restrict__ xs, int64_t nq_pad, const float4 *__restrict__ tquad, int64_t n,
              int64_t chunk, float *__restrict__ out) {
    pdl_enter();
    __shared__ __align__(16) float4 sm[RM_TS];
    const int64_t q0 = (int64_t)blockIdx.x * (2 * PP * RM_THREADS);
    float2 X[PP][3], m[PP];
#pragma unroll
    for (int pp = 0; pp < PP; ++pp) {
        const int64_t q = q0 + 2 * (pp * RM_THREADS + threadIdx.x);
        for (int t = 0; t < 3; ++t)
            X[pp][t] = t < D ? *reinterpret_cast<const float2 *>(xs + t * nq_pad + q) : make_float2(0.f, 0.f);
        m[pp] = make_float2(-INFINITY, -INFINITY);
    }
    const int64_t c_begin = (int64_t)blockIdx.y * chunk, c_end = min(n, c_begin + chunk);
    for (int64_t t0 = c_begin; t0 < c_end; t0 += RM_TS) {
        const int cnt = (int)min((int64_t)RM_TS, c_end - t0);
        __syncthreads();
        for (int i = threadIdx.x; i < cnt; i += RM_THREADS) sm[i] = tquad[t0 + i];
        if ((cnt & 1) && threadIdx.x == 0) sm[cnt] = tquad[t0 + cnt - 1];   // cnt < RM_TS: in range
        __syncthreads();
#pragma unroll 4
        for (int i = 0; i < cnt; i += 2) {
            const float4 w0 = sm[i], w1 = sm[i + 1];
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
                const float2 a = pair_exponent<D>(X[pp], w0), b = pair_exponent<D>(X[pp], w1);
                m[pp].x = max3f(m[pp].x, a.x, b.x);
                m[pp].y = max3f(m[pp].y, a.y, b.y);
            }
        }
    }
#pragma unroll
    for (int pp = 0; pp < PP; ++pp) {
        const int64_t q = q0 + 2 * (pp * RM_THREADS + threadIdx.x);
        *reinterpret_cast<float2 *>(out + (int64_t)blockIdx.y * nq_pad + q) = m[pp];
    }
}

__device__ __forceinline__ void block_max_key(float v, unsigned *key) {
    __shared__ float sh[32];
    v = warp_max_f(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = fmaxf(v, sh[w]);
        if (v > -INFINITY) atomicMax(key, ordered_key(v));
    }
}

// Per point: max_j r_qj, the row record (x', max - t1), A_q = k |x'|^2 - max;
// per target: the row record (w, log2(nu / sum m) - 60 - c) and B_j.  The
// largest A_q, B_j and |B_j| go into the result block.
__global__ void k_skip_operands(const float *__restrict__ part, int k1, int64_t nq_pad, int64_t nq,
                                const float *__restrict__ xs, const double *__restrict__ x64, int d,
                                double kappa, float t1, const double *__restrict__ psi, double eps,
                                const double *__restrict__ nu, double msum, int64_t n, int64_t n_pad,
                                const float4 *__restrict__ tquad, float4 *__restrict__ ptrow,
                                float *__restrict__ ptA, float4 *__restrict__ tgrow,
                                float *__restrict__ tgB, EvalResult *__restrict__ res) {
    pdl_enter();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float amax = -INFINITY, bmax = -INFINITY, babs = -INFINITY;
    // points or targets per block (blockIdx.y): a thread's FP64 chains would add up
    if (blockIdx.y == 0 && i < nq_pad) {
        float4 row = make_float4(0.f, 0.f, 0.f, INFINITY);
        float A = -INFINITY;
        if (i < nq) {
            float mx = -INFINITY;
            for (int k = 0; k < k1; ++k) mx = fmaxf(mx, part[(int64_t)k * nq_pad + i]);
            float x[3] = {0.f, 0.f, 0.f};
            double r2 = 0.0;
            for (int t = 0; t < d; ++t) {
                x[t] = xs[t * nq_pad + i];
                r2 = fma(x64[i * d + t], x64[i * d + t], r2);
            }
            A = amax = (float)(kappa * r2 - (double)mx);
            row = make_float4(x[0], x[1], x[2], mx - t1);
        }
        ptrow[i] = row;
        ptA[i] = A;
    }
    if (blockIdx.y == 1 && i < n_pad) {
        float4 r = tquad[i];
        float B = -INFINITY;
        r.w = INFINITY;
        if (i < n) {
            double bh, bl;
            target_B(psi[i], psi[0], eps, nu[i], bh, bl);
            B = bmax = (float)bh;
            babs = fabsf(B);
            r.w = (float)(log2(nu[i] / msum) - 60.0) - tquad[i].w;
        }
        tgrow[i] = r;
        tgB[i] = B;
    }
    if (blockIdx.y == 0) {
        block_max_key(amax, &res->fx_key[0]);
    } else {
        block_max_key(bmax, &res->fx_key[1]);
        block_max_key(babs, &res->fx_key[2]);
    }
}

// Order of the target rows of pass 2: by cells of a 2^b grid in Morton order, so
// that a warp's targets are near each other and most of a far point's pairs are
// skipped by whole warps: at eps 1e-3 (98,304 x 16,384) the FP64 pass 2 takes 1.6
// ms, 3.7 in the caller's order.  Which rows share a warp decides which columns
// below 2^-60 of a sum enter it in the compensated and mixed passes, so the order is
// a function of the data: a stable counting sort, once per problem.  Chunks of
// rows count their cells (k_cell_count), a cell's counts are summed over the chunks
// (k_cell_chunks) and the cells (k_cell_scan), and one warp of each chunk's block places
// its rows in their order (k_cell_scatter).
__global__ void __launch_bounds__(SORT_THREADS)
    k_cell_count(const double *__restrict__ pos, int64_t n, int64_t rows, int step, int d, double half,
                 int *__restrict__ cell, int *__restrict__ hist) {
    __shared__ int cnt[SORT_CELLS];
    for (int i = threadIdx.x; i < SORT_CELLS; i += SORT_THREADS) cnt[i] = 0;
    __syncthreads();
    const int64_t j0 = (int64_t)blockIdx.x * rows, j1 = min(n, j0 + rows);
    const int bits = d == 3 ? 4 : 6;
    for (int64_t j = j0 + threadIdx.x; j < j1; j += SORT_THREADS) {
        int id = 0;
        for (int t = 0; t < d; ++t) {
            const double u = half > 0.0 ? (pos[j * step * d + t] / half + 1.0) * 0.5 : 0.0;
            const int c = min(max((int)(u * (1 << bits)), 0), (1 << bits) - 1);
            for (int b = 0; b < bits; ++b) id |= ((c >> b) & 1) << (d * b + t);
        }
        cell[j] = id;
        atomicAdd(&cnt[id], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SORT_CELLS; i += SORT_THREADS) hist[(int64_t)blockIdx.x * SORT_CELLS + i] = cnt[i];
}

// a cell's counts become its rows in the chunks before; total: all of its rows
__global__ void k_cell_chunks(int *__restrict__ hist, int chunks, int *__restrict__ total) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    int sum = 0;
    for (int b0 = 0; b0 < chunks; b0 += 16) {
        int v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = b0 + i < chunks ? hist[(int64_t)(b0 + i) * SORT_CELLS + id] : 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (b0 + i < chunks) hist[(int64_t)(b0 + i) * SORT_CELLS + id] = sum;
            sum += v[i];
        }
    }
    total[id] = sum;
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

__global__ void __launch_bounds__(SORT_THREADS)
    k_cell_scatter(const int *__restrict__ cell, int64_t n, int64_t n_pad, int64_t rows,
                   const int *__restrict__ hist, const int *__restrict__ base, int *__restrict__ perm) {
    __shared__ int next[SORT_CELLS], ids[1024];
    const int tid = threadIdx.x, lane = tid & 31;
#pragma unroll 4
    for (int i = tid; i < SORT_CELLS; i += SORT_THREADS) next[i] = base[i] + hist[(int64_t)blockIdx.x * SORT_CELLS + i];
    const int64_t j0 = (int64_t)blockIdx.x * rows, j1 = min(n, j0 + rows);
    for (int64_t t0 = j0; t0 < j1; t0 += 1024) {
        const int cnt = (int)min((int64_t)1024, j1 - t0);
        __syncthreads();
        for (int i = tid; i < cnt; i += SORT_THREADS) ids[i] = cell[t0 + i];
        __syncthreads();
        if (tid < 32)
            for (int g = 0; g < cnt; g += 32) {
                const bool in = g + lane < cnt;
                const int id = in ? ids[g + lane] : SORT_CELLS;
                const unsigned same = __match_any_sync(0xffffffffu, id);
                const int rank = __popc(same & ((1u << lane) - 1u));
                if (in) perm[next[id] + rank] = (int)(t0 + g + lane);
                __syncwarp();
                if (in && rank == 0) next[id] += __popc(same);
                __syncwarp();
            }
    }
    for (int64_t j = n + (int64_t)blockIdx.x * SORT_THREADS + tid; j < n_pad; j += (int64_t)gridDim.x * SORT_THREADS)
        perm[j] = (int)j;
}

// The same maxima where the work is large: a warp holds 256 neighbouring points (by
// pairs, in the order of perm), tests 32 targets at a time against their box and
// takes those that may exceed a point's maximum so far, with the margin of the FP32
// exponents: after the first targets those are few.  98,304 x 65,536 at eps 1e-3:
// 765 -> 155 us; 98,304 x 16,384 at 1e-2: 201 -> 72.  Below 1e9 pairs the plain
// form is as fast.
template <int D>
__global__ void __launch_bounds__(RM_THREADS)
    k_row_max_skip(const float *__restrict__ xs, const int *__restrict__ perm, int64_t nq, int64_t nq_pad,
                   const float4 *__restrict__ tquad, int64_t n, int64_t chunk, float k, float kdiam2,
                   float *__restrict__ out) {
    pdl_enter();
    constexpr int PP = 4;
    __shared__ __align__(16) float4 s_t[RM_THREADS / 32][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float4 *const T = s_t[warp];
    const int64_t i0 = ((int64_t)blockIdx.x * (RM_THREADS / 32) + warp) * (32 * PP);   // point pairs
    const float inv4k = 0.25f / k;
    int q[PP];
    float2 X[PP][3], m[PP], kr2[PP];   // k |x|^2; -inf: no point
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int pp = 0; pp < PP; ++pp) {
        q[pp] = 2 * perm[i0 + 32 * pp + lane];
        float2 r2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            X[pp][t] = t < D ? *reinterpret_cast<const float2 *>(xs + t * nq_pad + q[pp]) : make_float2(0.f, 0.f);
            r2.x = fmaf(X[pp][t].x, X[pp][t].x, r2.x);
            r2.y = fmaf(X[pp][t].y, X[pp][t].y, r2.y);
            if (q[pp] < nq) lo[t] = fminf(lo[t], X[pp][t].x), hi[t] = fmaxf(hi[t], X[pp][t].x);
            if (q[pp] + 1 < nq) lo[t] = fminf(lo[t], X[pp][t].y), hi[t] = fmaxf(hi[t], X[pp][t].y);
        }
        kr2[pp] = make_float2(q[pp] < nq ? k * r2.x : -INFINITY, q[pp] + 1 < nq ? k * r2.y : -INFINITY);
        m[pp] = make_float2(-INFINITY, -INFINITY);
    }
    const Box box = make_box<D>(lo, hi, 2.f * k, inv4k);
    const int64_t c_begin = (int64_t)blockIdx.y * chunk, c_end = min(n, c_begin + chunk);
    const auto load = [&](int64_t g) { return g + lane < c_end ? tquad[g + lane] : make_float4(0.f, 0.f, 0.f, kPadC); };
    float thr = -INFINITY;   // the first 32 targets are all taken
    float4 nxt = load(c_begin);
#pragma unroll 1
    for (int64_t g = c_begin; g < c_end; g += 32) {
        const float4 w = nxt;
        nxt = load(g + 32);
        __syncwarp();
        T[lane] = w;
        const float B = fmaf(fmaf(w.x, w.x, fmaf(w.y, w.y, w.z * w.z)), inv4k, w.w);
        const float bound = box_bound<D>(box, w, B) + 0x1p-19f * (fabsf(B) + kdiam2);
        unsigned need = __ballot_sync(0xffffffffu, bound >= thr);
        __syncwarp();
        if (!need) continue;
#pragma unroll 1
        for (; need; need &= need - 1) {
            const float4 v = T[__ffs(need) - 1];
#pragma unroll
            for (int pp = 0; pp < PP; ++pp) {
                const float2 a = pair_exponent<D>(X[pp], v);
                m[pp].x = fmaxf(m[pp].x, a.x);
                m[pp].y = fmaxf(m[pp].y, a.y);
            }
        }
        float V = -INFINITY;
#pragma unroll
        for (int pp = 0; pp < PP; ++pp) V = fmaxf(V, fmaxf(kr2[pp].x - m[pp].x, kr2[pp].y - m[pp].y));
        thr = -warp_max_f(V);
    }
#pragma unroll
    for (int pp = 0; pp < PP; ++pp)
        *reinterpret_cast<float2 *>(out + (int64_t)blockIdx.y * nq_pad + q[pp]) = m[pp];
}

template <int D>
void row_max(rsot_problem *p, double eps) {
    dim3 g((unsigned)(p->nq_pad / (2 * p->sk_pp * RM_THREADS)), (unsigned)p->sk_k);
    const float k = (float)(kLog2e / (2.0 * eps)), kd = (float)(kLog2e / (2.0 * eps) * p->diam2);
    const bool over = overlap_pass(g, prep_blocks(p), p->num_sms, 0);
    if (p->sk_perm_q)
        launch_pdl(over, k_row_max_skip<D>, g, RM_THREADS, 0, p->stream, p->xs, p->sk_perm_q,
                   p->nq, p->nq_pad, p->tquad, p->n, p->sk_chunk, k, kd, p->sk_part);
    else
        launch_pdl(over, p->sk_pp == 4 ? k_row_max<D, 4> : k_row_max<D, 1>, g, RM_THREADS, 0,
                   p->stream, p->xs, p->nq_pad, p->tquad, p->n, p->sk_chunk, p->sk_part);
}

}  // namespace

// the smallest column split whose CTAs fill the resident slots (at most 5 % idle
// in the last wave); where a CTA per tile does not fill them, that, up to 64 splits (of
// few row blocks one more split fills hardly more slots, and there was none: compensated
// 1,000 x 1,000 173 -> 94 us, 64 x 2,000 266 -> 100; more partials than 64 cost what the
// shorter passes save, 1,000 x 65,536 with 256: 291 -> 331)
int split_for_slots(int64_t units, int64_t tiles, int64_t slots) {
    const int64_t least = units * tiles <= slots ? std::min<int64_t>(tiles, 64) : 1;
    int best = (int)least;
    double best_eff = least > 1 ? (double)(units * least) / (double)slots : 0.0;
    for (int64_t s = least; s <= std::min<int64_t>(tiles, 256); ++s) {
        const int64_t items = units * s, waves = (items + slots - 1) / slots;
        const double eff = (double)items / (double)(waves * slots);
        if (eff > best_eff + 0.01) best_eff = eff, best = (int)s;
        if (items >= slots && eff >= 0.95) return (int)s;
    }
    return best;
}

void skip_free(rsot_problem *p) {
    cudaFree(p->sk_buf);
    p->sk_buf = nullptr;
}

// Chunks of rows: counting and placing 1,024 rows take 10 us each, a chunk's counts 0.1 us
// of k_cell_chunks (sorting 16,384 rows 35 us with 16 chunks, 13 without the stable order).
static int64_t sort_chunks(int64_t n) {
    return std::max<int64_t>(1, std::min<int64_t>(512, (int64_t)sqrt((double)n / 5.0)));
}

size_t cell_order_scratch(int64_t n) { return ((size_t)n + (size_t)(sort_chunks(n) + 1) * SORT_CELLS) * sizeof(int); }

cudaError_t cell_order(rsot_problem *p, const double *pos, int64_t n, int64_t n_pad, int *perm, void *scratch,
                       int step) {
    const int64_t chunks = sort_chunks(n), rows = (n + chunks - 1) / chunks;
    int *const total = static_cast<int *>(scratch), *const hist = total + SORT_CELLS,
               *const cell = hist + chunks * SORT_CELLS;
    k_cell_count<<<(unsigned)chunks, SORT_THREADS, 0, p->stream>>>(pos, n, rows, step, p->d, p->half_ext, cell, hist);
    k_cell_chunks<<<SORT_CELLS / 64, 64, 0, p->stream>>>(hist, (int)chunks, total);
    k_cell_scan<<<1, 1024, 0, p->stream>>>(total);
    k_cell_scatter<<<(unsigned)chunks, SORT_THREADS, 0, p->stream>>>(cell, n, n_pad, rows, hist, total, perm);
    return cudaGetLastError();
}

// The estimates of the pair skipping work on squared distances, on k and on weights
// in FP32, here and in rsot_mskip.cu: units of length in which these leave its range,
// or so nearly that a squared length of 1e-6 of the data's does, take the passes
// without them.
bool skip_estimate_fits(const rsot_problem *p, double kappa) {
    return (p->diam2 == 0.0 || (p->diam2 >= 0x1p-64 && p->diam2 <= 0x1p100)) && kappa >= 0x1p-90 && kappa <= 0x1p88 &&
           p->nu_max <= 0x1p127;
}

// buffers and the target order, once per problem; false: not for these sizes,
// or no memory (the callers have passes that need none of it)
bool skip_ready(rsot_problem *p, double eps) {
    const double kappa = kLog2e / (2.0 * eps);
    // the estimate's error bound must allow a decision
    if (!(kappa * p->diam2 <= 0x1p23) || !skip_estimate_fits(p, kappa) || !(p->msum > 0.0)) return false;
    if (p->sk_buf) return true;
    const int64_t tiles = (p->n + RM_TS - 1) / RM_TS;
    p->sk_pp = p->nq_pad / 1024 * tiles >= 4 * p->num_sms ? 4 : 1;
    // also the chunks of the compensated pass 1, whose work skipping leaves uneven
    // (98,304 x 65,536: 2.06 ms with 6 CTAs per SM, 1.95 with 24)
    p->sk_k = split_for_slots(p->nq_pad / (2 * p->sk_pp * RM_THREADS), tiles, (int64_t)p->num_sms * 24);
    p->sk_chunk = (tiles + p->sk_k - 1) / p->sk_k * RM_TS;
    p->sk_k = (int)((p->n + p->sk_chunk - 1) / p->sk_chunk);
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t np = (size_t)p->nq_pad, nt = (size_t)p->n_pad;
    const bool skip_max = p->sk_pp == 4 && (double)p->nq * (double)p->n >= 1e9;   // k_row_max_skip
    const size_t o_perm = take(nt * 4), o_pq = take(skip_max ? np / 2 * 4 : 0);
    const size_t o_part = take(np * 4 * p->sk_k), o_prow = take(np * 16), o_pcol = take(np * 16);
    const size_t o_pA = take(np * 4), o_trow = take(nt * 16), o_tB = take(nt * 4);
    // while the orders are made, all that follows them is scratch
    at = std::max(at, o_part + std::max(cell_order_scratch(p->n), cell_order_scratch((p->nq + 1) / 2)));
    // in steps of 256 KiB, of which the allocator more often has a block left from a handle
    // before (24,576 x 512 in a loop of new handles: cudaMalloc 77 -> 5 us)
    at = (at + 262143) / 262144 * 262144;
    char *b = nullptr;
    if (cudaMalloc(&b, at) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    p->sk_buf = b;
    p->sk_part = reinterpret_cast<float *>(b + o_part);
    p->sk_ptrow = reinterpret_cast<float4 *>(b + o_prow);
    p->sk_ptcol = reinterpret_cast<float4 *>(b + o_pcol);
    p->sk_ptA = reinterpret_cast<float *>(b + o_pA);
    p->sk_tgrow = reinterpret_cast<float4 *>(b + o_trow);
    p->sk_tgB = reinterpret_cast<float *>(b + o_tB);
    p->sk_perm = reinterpret_cast<int *>(b + o_perm);
    p->sk_perm_q = skip_max ? reinterpret_cast<int *>(b + o_pq) : nullptr;
    cudaError_t e = cell_order(p, p->y64, p->n, p->n_pad, p->sk_perm, b + o_part);
    if (!e && skip_max) e = cell_order(p, p->x64, (p->nq + 1) / 2, p->nq_pad / 2, p->sk_perm_q, b + o_part, 2);
    // once per problem: a later evaluation may run on another stream
    if (e || cudaStreamSynchronize(p->stream) != cudaSuccess) {
        cudaGetLastError();
        skip_free(p);
        return false;
    }
    return true;
}

double skip_t1(const rsot_problem *p) { return 60.0 + log2((double)p->n) + 1.0; }

cudaError_t launch_skip(rsot_problem *p, const double *psi, double eps) {
    cudaStream_t st = p->stream;
    cudaError_t e = launch_prep_mixed(p, psi, eps);
    if (e) return e;
    trace_begin(p, "row_max");
    (p->d == 3 ? row_max<3> : row_max<2>)(p, eps);
    trace_end(p);
    const int64_t most = std::max(p->nq_pad, p->n_pad);
    const unsigned t = small_threads(most, p->num_sms);
    trace_begin(p, "skip_operands");
    launch_pdl(true, k_skip_operands, dim3((unsigned)(most / t), 2), t, 0, st, p->sk_part, p->sk_k, p->nq_pad, p->nq, p->xs, p->x64, p->d,
                                        kLog2e / (2.0 * eps), (float)skip_t1(p), psi, eps, p->nu, p->msum,
                                        p->n, p->n_pad, p->tquad, p->sk_ptrow, p->sk_ptA, p->sk_tgrow,
                                        p->sk_tgB, p->res_dev);
    trace_end(p);
    return cudaGetLastError();
}

}  // namespace rsot
