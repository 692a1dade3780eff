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
//     unit, together close to 1, are added to the columns' constants).  F is
//     at most 52 and falls by two for every factor 4 of the largest exponent
//     that occurs, whose FP64 rounding grows alike.
//   * The exponent n = kappa d^2 - C (C: the column's constant, 64-bit, modulo
//     2^(64-F)) gives 2^-n = 2^-I T[i] q: I its integer part, T[i] = 2^(-i/2048)
//     from the next 11 bits (table of FP64 values), and q = 2^-g, g < 2^-11, as
//     1 - z + z^2/2 (1 - c z), z = g ln 2, in 32-bit integer multiplications
//     (c is 1/3 less the value that centres the dropped z^4/24: error below
//     2^-54); its FP64 bits are those of 1.0 minus the integer 2^53 (1 - q).
//   * A term of pass 2 is m_q p_qj, and the exponent field of its FP64 value has no
//     lower end to stop at, so every term that is summed has to stay above 2^-1020:
//     points whose mass is below 2^-61 of the smallest weight over their number are
//     left out of pass 2 (all of them together stay below 2^-61 nu_j), which bounds
//     the others from below by the weights (fx_exponents_fit).
//   * Pairs that cannot change a sum by 2^-60 of it are skipped (rsot_skip.cuh).
//     The wrapped integers are only read for pairs that are not, whose exponents
//     lie inside the range that F allows.
// Error of an exponent: about 2^-F (F = 52: 2.2e-16) against about 2^-53 of the
// largest of kappa d^2, B_j in the FP64 passes.
//
// Where the skipping's estimate could be off by more than 16 or the exponents
// need F < 46 the records kernel raises kErrRange64 and the caller runs the FP64
// passes; they also run where the weights reach further down than that allows.
//
// A pair and pass takes about 55 instructions: the FP64 pipe (one fma) is 63 %
// busy, the FMA pipe with the multiplications 76 %.
#include <math.h>

#include <algorithm>

#include "rsot_internal.cuh"
#include "rsot_exp64.cuh"
#include "rsot_skip.cuh"

namespace rsot {

// integer operand record: (h0, l0, h1, l1), (h2, l2, -C low, -C high)
struct FxRec {
    int4 a, b;
};

namespace {

constexpr int FX_THREADS = 128;
constexpr int FX_TS = 64;         // columns per shared-memory tile
constexpr int FX_TAB = 2048;      // 2^(-i/2048)
constexpr int FX_U = 4;           // columns at once where a thread has one row (24,576 x 512,
                                  // with tiles of 128 columns: 63, 55, 47 us a pass for 1, 2, 4;
                                  // 41 with tiles of 64, half the chain of a CTA)
constexpr int FX_FMAX = 52, FX_FMIN = 46;

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

// Integer operands, the fraction bits F from the ranges, the integral shifts of
// the rows and the table of 2^(-i/2048).
__global__ void k_fx_records(const double *__restrict__ x64, int64_t nq, int64_t nq_pad,
                             const double *__restrict__ y64, int64_t n, int64_t n_pad, int d,
                             double c0, double c1, double kappa_diam2, double tmax,
                             const double *__restrict__ psi, double eps,
                             const double *__restrict__ nu, const float *__restrict__ ptA,
                             FxRec *__restrict__ prec, int *__restrict__ ptshift,
                             FxRec *__restrict__ trec, int *__restrict__ tgshift,
                             double *__restrict__ tgscale, double *__restrict__ tab,
                             EvalResult *__restrict__ res) {
    pdl_enter();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double amax = from_key(res->fx_key[0]), bmax = from_key(res->fx_key[1]);
    const double E = skip_error(res, (float)kappa_diam2);
    const double L = (bmax + amax + tmax + 4.0 * E + 4.0) / 0.9;   // largest kappa d^2 of a kept pair
    int F = FX_FMAX;
    while (F >= FX_FMIN && L >= ldexp(1.0, 62 - F)) F -= 2;
    const bool bad = F < FX_FMIN || !(E <= 16.0) || !(L > 0.0);
    if (bad) F = FX_FMIN;
    if (i == 0) {
        res->fx_F = F;
        if (bad) atomicOr(&res->flags, kErrRange64);
    }
    const int s = (F + 62) / 2;
    if (bad) return;
    // one part per block (blockIdx.y): a thread's chains of FP64 would add up
    if (blockIdx.y == 0 && i < nq_pad) {
        int2 c[3] = {};
        if (i < nq)
            for (int t = 0; t < d; ++t) c[t] = fx_coord(x64[i * d + t], c0, c1, s);
        FxRec r;
        r.a = make_int4(c[0].x, c[0].y, c[1].x, c[1].y);
        r.b = make_int4(c[2].x, c[2].y, 0, 0);
        prec[i] = r;
        ptshift[i] = i < nq ? -(int)rintf(ptA[i]) : 0;   // the point's largest exponent
    }
    if (blockIdx.y == 1 && i < n_pad) {
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
        tgshift[i] = -sh;
        tgscale[i] = scale;
    }
    if (blockIdx.y == 2 && i < FX_TAB) {
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

// rows and columns of a pass: integer records, FP32 records, values of the ball
// test (rsot_skip.cuh) and the factors that turn the FP32 records into positions
struct FxRows {
    const FxRec *rec;
    const float4 *f;
    const float *val;
    const int *shift;   // integral, added to the exponent's negative
    const int *perm;    // row order (null: as stored)
    bool pairs;         // of pairs of rows
    float slack;        // added to val in the ball test
    float scale;
    int64_t count, pad;
};
struct FxCols {
    const FxRec *rec;
    const float4 *f;
    const float *val;
    float scale;
    int64_t count;
};

// ----------------------------------------------------------------------------
// One pass: out[chunk][row] = sum over the chunk's columns of
// 2^(C_col - kappa d^2 - shift_row).  Pass 1: rows = points, columns = targets;
// pass 2: rows = targets (in the order of perm), columns = points.
// ----------------------------------------------------------------------------
// the pair's FP32 exponent reaches the row's threshold
template <int D>
__device__ __forceinline__ bool pair_on(const float4 &f, const float4 &x) {
    float e = f.w;
    if (D == 3) e = fmaf(f.z, x.z, e);
    e = fmaf(f.x, x.x, fmaf(f.y, x.y, e));
    return e >= x.w;
}

// 2^(C_col - kappa d^2 - shift_row) = Ts q
template <int D>
__device__ __forceinline__ void fx_term(const FxRec &rec, const int (&H)[3], const int (&Lo)[3], int rs, int shE,
                                        int shI, int shG, const double *s_tab, double &Ts, double &q) {
    const int4 a = rec.a, b = rec.b;
    const long long nc = (long long)(((unsigned long long)(unsigned)b.w << 32) | (unsigned)b.z);
    const int h0 = H[0] - a.x, h1 = H[1] - a.z;
    const int l0 = Lo[0] - a.y, l1 = Lo[1] - a.w;
    long long hh = (long long)h0 * h0 + nc;
    long long mid = (long long)h0 * l0;
    hh += (long long)h1 * h1;
    mid += (long long)h1 * l1;
    if (D == 3) {
        const int h2 = H[2] - b.x, l2 = Lo[2] - b.y;
        hh += (long long)h2 * h2;
        mid += (long long)h2 * l2;
    }
    hh += mid >> 30;
    const unsigned lo = (unsigned)hh;
    const int hi = (int)(hh >> 32) + rs;
    const int ex = hi >> shE;                       // integer part
    const unsigned off = ((unsigned)hi >> shI) & ((FX_TAB - 1u) << 3);
    const double T = *reinterpret_cast<const double *>(reinterpret_cast<const char *>(s_tab) + off);
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
    q = __longlong_as_double(0x3FF0000000000000ll - (long long)(z >> 22));
    Ts = __hiloint2double(__double2hiint(T) - (ex << 20), __double2loint(T));
}

template <int D, int R>
__global__ void __launch_bounds__(FX_THREADS)
    k_fx_pass(FxRows rows, FxCols cols, int64_t chunk, float kappa, float kdiam2,
              const double *__restrict__ tab, double *__restrict__ out,
              const EvalResult *__restrict__ res) {
    pdl_enter();
    if (res->flags & kErrRange64) return;
    __shared__ __align__(16) FxRec s_rec[FX_TS];
    __shared__ __align__(16) float4 s_f[FX_TS];
    __shared__ float s_v[FX_TS];
    __shared__ double s_tab[FX_TAB];
    const int tid = threadIdx.x, lane = tid & 31;
    for (int i = tid; i < FX_TAB / 2; i += FX_THREADS)
        reinterpret_cast<double2 *>(s_tab)[i] = reinterpret_cast<const double2 *>(tab)[i];
    const int F = res->fx_F;
    const float margin = 2.0f * skip_error(res, kdiam2);
    const int shE = F - 32, shI = F - 46, shG = 75 - F;
    int H[R][3], Lo[R][3], rs[R], at[R];
    float4 xf[R];
    float val[R];
    double acc[R];
    constexpr int U = FX_U;
#pragma unroll
    for (int k = 0; k < R; ++k) {
        const int64_t i = (int64_t)blockIdx.x * (FX_THREADS * R) + R * tid + k;
        acc[k] = 0.0;
        xf[k] = make_float4(0.f, 0.f, 0.f, INFINITY);
        val[k] = -INFINITY;
        rs[k] = 0;
        at[k] = -1;
        FxRec r;
        r.a = r.b = make_int4(0, 0, 0, 0);
        int64_t a = i;   // a pair's second row may be padding
        if (rows.perm && rows.pairs && (i & ~(int64_t)1) < rows.count) a = 2 * rows.perm[i >> 1] + (i & 1);
        else if (rows.perm && i < rows.count) a = rows.perm[i];
        if (a < rows.count) {
            at[k] = (int)a;
            r = rows.rec[at[k]];
            xf[k] = rows.f[at[k]];
            xf[k].w -= margin;
            val[k] = rows.val[at[k]] + rows.slack + margin;
            rs[k] = (int)((unsigned)rows.shift[at[k]] << shE);
        }
        H[k][0] = r.a.x, Lo[k][0] = r.a.y;
        H[k][1] = r.a.z, Lo[k][1] = r.a.w;
        H[k][2] = r.b.x, Lo[k][2] = r.b.y;
    }
    // where k diam^2 is a few times the depth of the sums, few columns are skipped
    // whole: the pair test alone (24,576 x 512, eps 1e-2, one column at a time: 51 us
    // a pass, 63 with)
    const bool use_ball = kdiam2 > 4.0f * rows.slack;
    RowBall ball = {};
    if (use_ball) ball = row_ball(xf[0], val[0], xf[R - 1], val[R - 1], rows.scale);
    const int64_t c_begin = (int64_t)blockIdx.y * chunk;
    const int64_t c_end = min(cols.count, c_begin + chunk);
    for (int64_t t0 = c_begin; t0 < c_end; t0 += FX_TS) {
        const int cnt = (int)min((int64_t)FX_TS, c_end - t0);
        __syncthreads();
        if (tid < cnt) {
            s_rec[tid] = cols.rec[t0 + tid];
            s_f[tid] = cols.f[t0 + tid];
            s_v[tid] = cols.val[t0 + tid];
        }
        __syncthreads();
        for (int g = 0; g < cnt; g += 32) {
            unsigned need = __ballot_sync(
                0xffffffffu, g + lane < cnt && (!use_ball || ball_needs(ball, s_f[g + lane], s_v[g + lane],
                                                                        cols.scale, kappa)));
            if constexpr (R == 1) {
                // U columns at once, straight through for every lane of the warp:
                // the chain of one pair (about 330 cycles) overlaps the others'
                while (need) {
                    int c[U];
                    bool on[U];
                    unsigned any = 0;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const bool has = need != 0;
                        c[u] = has ? g + __ffs(need) - 1 : c[0];
                        need &= need - 1;
                        on[u] = has && pair_on<D>(s_f[c[u]], xf[0]);
                        any |= on[u];
                    }
                    if (!__any_sync(0xffffffffu, any)) continue;
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        double Ts, q;
                        fx_term<D>(s_rec[c[u]], H[0], Lo[0], rs[0], shE, shI, shG, s_tab, Ts, q);
                        acc[0] = fma(on[u] ? Ts : 0.0, q, acc[0]);
                    }
                }
            } else {
                for (; need; need &= need - 1) {
                    const int c = g + __ffs(need) - 1;
                    const float4 f = s_f[c];
                    const FxRec rec = s_rec[c];
#pragma unroll
                    for (int k = 0; k < R; ++k) {
                        if (!pair_on<D>(f, xf[k])) continue;
                        double Ts, q;
                        fx_term<D>(rec, H[k], Lo[k], rs[k], shE, shI, shG, s_tab, Ts, q);
                        acc[k] = fma(Ts, q, acc[k]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < R; ++k)
        if (at[k] >= 0) out[(int64_t)blockIdx.y * rows.pad + at[k]] = acc[k];
}

// Per point: L_q, the mass's J term, and, for masses from m_least on, the column of
// pass 2: u_q = log2(m_q / S_q) - shift_q, (x', -R_q) and A_q.
__global__ void k_fx_combine(const double *__restrict__ part, int k1, int64_t nq, int64_t nq_pad,
                             const int *__restrict__ shift, const double *__restrict__ mass,
                             double m_least, const double *__restrict__ psi, double eps, float t1,
                             const float4 *__restrict__ ptrow, FxRec *__restrict__ prec,
                             float4 *__restrict__ ptcol, float *__restrict__ ptA,
                             double *__restrict__ lse_buf, double *__restrict__ blockJ,
                             const EvalResult *__restrict__ res) {
    pdl_enter();
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
        const float4 x = ptrow[q];
        const float rise = (float)M + ptA[q] + __log2f((float)S);   // R_q - max_j r_qj
        float4 col = make_float4(x.x, x.y, x.z, kPadC);
        float A = -INFINITY;
        if (m > 0.0) contrib = m * (psi[0] + eps * L);
        if (m >= m_least) {
            int em, es;
            const double fm = log2_split(m, em), fs = log2_split(S, es);
            const long long C = 1 - to_fixed((double)(em - es - M), fm - fs, res->fx_F);
            prec[q].b.z = (int)(C & 0xffffffffll);
            prec[q].b.w = (int)(C >> 32);
            col.w = -(x.w + t1 + rise);
            A = ptA[q] - rise;
        }
        ptcol[q] = col;
        ptA[q] = A;
    }
    store_partial(contrib, blockJ);
}

// rows per thread: 2 share a column's loads, 1 where that leaves SMs idle
inline int fx_rows(const rsot_problem *p, int64_t rows, int64_t cols) {
    return rows / (2 * FX_THREADS) * (cols / 512) >= 5 * p->num_sms ? 2 : 1;
}

template <int D>
void fx_launch(rsot_problem *p, int R, const FxRows &rows, const FxCols &cols, int64_t chunk, int splits,
               double eps, double *out, int64_t before) {
    const float kappa = (float)(kLog2e / (2.0 * eps)), kd = (float)(kLog2e / (2.0 * eps) * p->diam2);
    // blocks of padding rows alone are not launched
    dim3 g((unsigned)((rows.count + FX_THREADS * R - 1) / (FX_THREADS * R)), (unsigned)splits);
    launch_pdl(overlap_pass(g, before, p->num_sms, p->num_sms / 2), R == 2 ? k_fx_pass<D, 2> : k_fx_pass<D, 1>, g, FX_THREADS, 0, p->stream,
               rows, cols, chunk, kappa, kd, p->fx_tab, out, p->res_dev);
}

// buffers of the fixed-point passes, once per problem; false: no memory (the
// FP64 passes need none of them)
bool fx_alloc(rsot_problem *p) {
    if (p->fx_buf) return true;
    auto chunked = [&](int64_t rows, int64_t cols, int &split, int64_t &chunk) {
        const int64_t blk = FX_THREADS * fx_rows(p, rows, cols), tiles = (cols + FX_TS - 1) / FX_TS;
        // about 60 CTAs per SM: skipped columns leave their work uneven (98,304 x
        // 16,384: 8.9 ms with 5 per SM, 8.8 with 20, 8.4 with 60, 8.3 with 100; 61,206 x
        // 5,003: 1.69, 1.58, 1.55, 1.55); 256 splits bound the last kernel's sums
        const int64_t units = (rows + blk - 1) / blk;
        const int64_t s = std::min({tiles, (60 * p->num_sms + units - 1) / units, (int64_t)256});
        chunk = (tiles + s - 1) / s * FX_TS;
        split = (int)((cols + chunk - 1) / chunk);
    };
    chunked(p->nq, p->n, p->fx_k1, p->fx_chunk1);
    chunked(p->n, p->nq, p->fx_s2, p->fx_chunk2);
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t o = at;
        at += (bytes + 255) / 256 * 256;
        return o;
    };
    const size_t np = (size_t)p->nq_pad, nt = (size_t)p->n_pad;
    const size_t o_prec = take(np * sizeof(FxRec)), o_trec = take(nt * sizeof(FxRec));
    const size_t o_psh = take(np * 4), o_tsh = take(nt * 4), o_tsc = take(nt * 8);
    const size_t o_tab = take(FX_TAB * 8), o_p1 = take(np * 8 * p->fx_k1), o_p2 = take(nt * 8 * p->fx_s2);
    char *b = nullptr;
    if (cudaMalloc(&b, at) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    p->fx_buf = b;
    p->fx_prec = reinterpret_cast<FxRec *>(b + o_prec);
    p->fx_trec = reinterpret_cast<FxRec *>(b + o_trec);
    p->fx_ptshift = reinterpret_cast<int *>(b + o_psh);
    p->fx_tgshift = reinterpret_cast<int *>(b + o_tsh);
    p->fx_tgscale = reinterpret_cast<double *>(b + o_tsc);
    p->fx_tab = reinterpret_cast<double *>(b + o_tab);
    p->fx_part1 = reinterpret_cast<double *>(b + o_p1);
    p->fx_part2 = reinterpret_cast<double *>(b + o_p2);
    return true;
}

}  // namespace

void fx64_free(rsot_problem *p) {
    cudaFree(p->fx_buf);
    p->fx_buf = nullptr;
}

// the smallest mass that takes part in pass 2
static double fx_least_mass(const rsot_problem *p) { return ldexp(p->nu_min, -61) / (double)p->nq; }

// A term of pass 2 that is summed is at least fx_least_mass() times the smallest p_qj
// of a pair that is kept, 2^-60 nu_j / sum m less four errors E <= 16 of the estimate:
// its exponent stays above -1020 (weights down to about 1e-120 of a total mass of 1).
static bool fx_exponents_fit(const rsot_problem *p) {
    return log2(fx_least_mass(p)) + (log2(p->nu_min) - log2(p->msum)) - 60.0 - 4.0 * 16.0 >= -1020.0;
}

bool fx64_ready(rsot_problem *p, double eps) {
    return fx_exponents_fit(p) && skip_ready(p, eps) && fx_alloc(p);
}

cudaError_t launch_dense_fx64(rsot_problem *p, const double *psi, double eps, double *grad) {
    cudaStream_t st = p->stream;
    const double kappa = kLog2e / (2.0 * eps);
    const float inv2k = (float)(0.5 / kappa);
    // sqrt(kappa) as c0 + c1: kappa = (1/eps) log2(e) / 2 in double-double
    const double inv = 1.0 / eps, inv_lo = -fma(inv, eps, -1.0) / eps;
    const double kh = inv * (0.5 * kLog2e);
    const double kl = fma(inv, 0.5 * kLog2e, -kh) + inv * (0.5 * 2.0355273740931033e-17) +
                      inv_lo * (0.5 * kLog2e);
    const double c0 = sqrt(kh), c1 = (-fma(c0, c0, -kh) + kl) / (2.0 * c0);
    const double t1 = skip_t1(p);
    const double tmax = std::max(t1, 60.0 + log2(p->msum / p->nu_min));   // largest slack of a row
    cudaError_t e = launch_skip(p, psi, eps);
    if (e) return e;
    const int64_t most = std::max({p->nq_pad, p->n_pad, (int64_t)FX_TAB});
    const unsigned tr = small_threads(most, p->num_sms);
    trace_begin(p, "fx_records");
    launch_pdl(
        true, k_fx_records, dim3((unsigned)(most / tr), 3), tr, 0, st, p->x64, p->nq, p->nq_pad, p->y64, p->n, p->n_pad, p->d, c0, c1, kappa * p->diam2, tmax, psi,
        eps, p->nu, p->sk_ptA, p->fx_prec, p->fx_ptshift, p->fx_trec, p->fx_tgshift, p->fx_tgscale,
        p->fx_tab, p->res_dev);
    trace_end(p);
    // compact warps where columns are skipped whole (use_ball)
    const int *const order = kappa * p->diam2 > 4.0 * t1 ? p->sk_perm_q : nullptr;
    const FxRows pts = {p->fx_prec, p->sk_ptrow, p->sk_ptA, p->fx_ptshift, order, true,
                        (float)t1,  1.f,         p->nq,     p->nq_pad};
    const FxCols tgt = {p->fx_trec, p->tquad, p->sk_tgB, inv2k, p->n};
    trace_begin(p, "fx_lse");
    (p->d == 3 ? fx_launch<3> : fx_launch<2>)(p, fx_rows(p, p->nq, p->n), pts, tgt, p->fx_chunk1, p->fx_k1,
                                              eps, p->fx_part1, 3 * (most / tr));
    trace_end(p);
    trace_begin(p, "fx_combine");
    const int nbq = (int)(p->nq_pad / 256);
    const unsigned tc = p->per_comb == 1 ? 256 : kSmall;
    launch_pdl(true, k_fx_combine, (unsigned)(p->nq_pad / tc), tc, 0, st, p->fx_part1, p->fx_k1, p->nq, p->nq_pad, p->fx_ptshift, p->mass,
                                      fx_least_mass(p), psi, eps, (float)t1, p->sk_ptrow, p->fx_prec, p->sk_ptcol,
                                      p->sk_ptA, p->lse_buf, p->blockJ, p->res_dev);
    trace_end(p);
    const FxRows tgr = {p->fx_trec,  p->sk_tgrow, p->sk_tgB, p->fx_tgshift, p->sk_perm, false,
                        (float)tmax, inv2k,       p->n,      p->n_pad};
    const FxCols ptc = {p->fx_prec, p->sk_ptcol, p->sk_ptA, 1.f, p->nq};
    trace_begin(p, "fx_grad");
    (p->d == 3 ? fx_launch<3> : fx_launch<2>)(p, fx_rows(p, p->n, p->nq), tgr, ptc, p->fx_chunk2, p->fx_s2,
                                              eps, p->fx_part2, p->nq_pad / tc);
    trace_end(p);
    return launch_finalize(p, psi, eps,
                           {p->fx_part2, p->fx_s2, p->n_pad, p->fx_tgscale, p->blockJ, nbq, p->per_comb, 0, p->per_prep},
                           grad);
}

}  // namespace rsot
