// The CG head on boxes of few elements, in double-float arithmetic on FP32
// pairs (df.cuh, ax_df_core.cuh): x += xa p, p = r + beta p, w = ax_e(p) and
// <w,p>_c.  Such solves run past convergence within the paper's fixed 100
// iterations, where CG amplifies the rounding of its operator to 1e-9 and more
// of x; with the arithmetic kept, their results stay what they were (the
// fixed-point operator is no less accurate).  On one CTA per SM and fewer it is
// also the faster head for most orders (df_head_elements).
//
// Thread layout ("line threads").  A CTA owns one element at a time and has
// 3 n^2 working threads: thread (d, a0, a1) owns one line of the element
// along direction d (r: (j,k); s: (i,k); t: (i,j)).  In the forward phase a
// thread loads its n inputs once from shared memory and produces the n
// derivative values of its line; the entries of D are compile-time indexed
// kernel parameters.  A pointwise phase contracts (wr, ws, wt) with the six
// geometric factors in place, the backward phase is the same line pattern with
// D^T, each direction writing its own partial array, and a final pointwise
// phase adds the three partials and writes w.
#include <math.h>

#include "ax_df_core.cuh"
#include "exact_sum.cuh"

namespace nekgb {

struct AxDfArgs {
    double *w;            // output (FP64, local storage)
    const double *r;      // residual
    double *p;            // search direction, updated in place
    double *x;            // iterate, receives the owed x += x_alpha p
    CgScalars *sc;
    double *partials;     // one <w,p> partial per CTA
    int dot_shift0;       // scale of the exact <w,p>_c sum (see launch_df_n)
    int dot_lim;          // a share of 2^dot_lim or more (scaled) may overflow the sum
    int finite;           // the operator's data (D and gxyz) has no NaN or Inf
    Mesh m;
    const float2 *g;      // gxyz pairs [E][6][n^3], scaled by 2^-(gexp-1023)
    int gexp;             // biased exponent of max|gxyz|
    int64_t E;
};

// v 2^S truncated toward zero to an integer, as a two's-complement 128-bit
// value.  The caller's S keeps |v| 2^S below 2^lim (lim = 125 - log2 of the
// number of shares, see the head), so no sum of shares overflows; a share
// that may reach 2^lim sets `out_of_range` (the solve then stops with a
// status instead of using a wrong sum).  The shift is clamped at 73; values
// whose scaled magnitude is below 1 give 0.
__device__ __forceinline__ u128 fixed_of(double v, int S, int lim, bool &out_of_range) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)((b >> 52) & 0x7ff);
    if (ex == 0) return 0;
    out_of_range |= ex - 1022 + S > lim;                 // |v| 2^S < 2^(ex - 1022 + S)
    const unsigned long long M = (b & 0xfffffffffffffull) | (1ull << 52);
    int sh = ex - 1075 + S;
    u128 mag;
    if (sh >= 0) {
        sh = sh > 73 ? 73 : sh;
        mag = (u128)M << sh;
    } else {
        mag = sh > -64 ? (u128)(M >> (-sh)) : (u128)0;
    }
    return (b >> 63) ? (u128)0 - mag : mag;
}

// The unpreconditioned two-kernel CG head with a software-pipelined,
// dynamically scheduled element loop.
//
// Scale.  The pairs of p are scaled by one power of two per iteration, 2^sh
// with sqrt(<p,p>_c) 2^sh in [1, 2) (<p,p>_c from the scalar block; every
// |p| is at most sqrt(8 <p,p>_c), as c >= 1/8), instead of a per-element
// maximum: that removes the exponent reduction and its barrier, and lets p
// be split straight from registers into shared memory.  Tiny entries lose
// low-order bits only below 2^-78 of that scale, far under the operator's
// rounding relative to max|w|.
//
// Pipeline.  The six shared arrays rotate roles between consecutive
// elements (X the input, F the three derivative arrays, P the partials):
//   even step: X = S0, F = (S1, S2, S3), P = (S0, S4, S5)
//   odd step:  X = S1, F = (S0, S2, S3), P = (S1, S4, S5)
// so the next element is staged into its X while the final pass reads the
// current P, which needs no barrier in between: four barriers per element.
//
// Schedule.  After its first element (blockIdx.x) a CTA takes the next one
// from a counter in the scalar block, so SMs that run slower take fewer
// elements (a static assignment left the slowest SM 12 % behind the mean).
// The counter is read at the start of a step and published just before the
// barrier that ends the backward pass, which hides the atomic's latency.
// <w,p>_c stays independent of the schedule because it is summed exactly:
// each thread's share of an element (its points' products, in a fixed
// order, in FP64) is converted to a 128-bit integer at the fixed scale 2^S
// (fixed_of, truncating) and added to the thread's integer sum; integer
// sums do not depend on the order of the additions.  The caller chooses S
// from <p,p>_c and a bound on the operator so that no sum can overflow
// (see launch_df_n); the result is rounded to FP64 once, at the end.
template <int N>
__device__ __forceinline__ u128 df_head_pipelined(const AxDfArgs &a, double beta, double xa, int S,
                                                  const DfEo<N> &D, float2 *sm,
                                                  bool &out_of_range) {
    constexpr int N2 = N * N, N3 = N * N * N;
    constexpr int T = ax_df_threads(N);
    __shared__ long long s_next;
    const int t = threadIdx.x;
    const double pn = a.sc->it == 0 ? a.sc->rr : a.sc->pn2;
    const int ep = (int)((__double_as_longlong(pn) >> 52) & 0x7ff);
    const int sh_in = ep == 0 ? 0 : -((ep - 1023) >> 1);
    const int sh_out = -sh_in + (a.gexp - 1023);
    float2 *S0 = sm, *S1 = sm + N3, *S2 = sm + 2 * N3, *S3 = sm + 3 * N3, *S4 = sm + 4 * N3, *S5 = sm + 5 * N3;
    constexpr int PPT = df_points_per_thread<N, T>();
    // x += xa p (the owed update), p = r + beta p, X = pairs of p 2^sh; the loads
    // of all of a thread's points are issued before the first store, which the
    // compiler could not do itself (a store might alias a later load)
    auto stage = [&](int64_t e, float2 *X) {
        const int64_t eb = e * N3;
        double *p = a.p + eb, *x = a.x + eb;
        const double *r = a.r + eb;
        double pv[PPT], rv[PPT], xv[PPT];
#pragma unroll
        for (int k = 0; k < PPT; k++) {
            const int q = t + k * T;
            if (q < N3) {
                pv[k] = p[q];
                rv[k] = r[q];
                if (xa != 0.0) xv[k] = __ldcs(x + q);
            }
        }
#pragma unroll
        for (int k = 0; k < PPT; k++) {
            const int q = t + k * T;
            if (q < N3) {
                if (xa != 0.0) __stcs(x + q, fma(xa, pv[k], xv[k]));
                const double v = fma(beta, pv[k], rv[k]);
                p[q] = v;
                X[q] = dfa::split_scaled<true>(v, sh_in);
            }
        }
    };
    // the box-face bits of this thread's points in the final pass, computed once
    FaceBits<N, T, PPT> pf;
    pf.init();
    u128 acc = 0;
    int64_t e = blockIdx.x;
    if (e < a.E) stage(e, S0);
    __syncthreads();
    for (int k = 0; e < a.E; k++) {
        const bool odd = k & 1;
        unsigned nxt = 0;
        if (t == 0) nxt = atomicAdd(&a.sc->next_elem, 1u);
        float2 *X = odd ? S1 : S0;
        float2 *F0 = odd ? S0 : S1;
        // forward: wr, ws, wt along this thread's line
        for (int task = t; task < 3 * N2; task += T) {
            int stride;
            const int base = line_of<N>(task, stride);
            float2 *Fd = task < N2 ? F0 : (task < 2 * N2 ? S2 : S3);
            line_eo<N>(X, Fd, base, stride, D.fwd);
        }
        __syncthreads();
        // geometric contraction, pointwise, in place
        const float2 *g = a.g + e * 6 * N3;
        for (int q = t; q < N3; q += T) {
            const float2 wr = F0[q], ws = S2[q], wt = S3[q];
            const float2 g0 = __ldcs(g + q), g1 = __ldcs(g + N3 + q), g2 = __ldcs(g + 2 * N3 + q);
            const float2 g3 = __ldcs(g + 3 * N3 + q), g4 = __ldcs(g + 4 * N3 + q), g5 = __ldcs(g + 5 * N3 + q);
            dfa::Acc ur = dfa::first(g0.x, g0.y, wr.x, wr.y);
            dfa::fma(ur, g1.x, g1.y, ws.x, ws.y);
            dfa::fma(ur, g2.x, g2.y, wt.x, wt.y);
            dfa::Acc us = dfa::first(g1.x, g1.y, wr.x, wr.y);
            dfa::fma(us, g3.x, g3.y, ws.x, ws.y);
            dfa::fma(us, g4.x, g4.y, wt.x, wt.y);
            dfa::Acc ut = dfa::first(g2.x, g2.y, wr.x, wr.y);
            dfa::fma(ut, g4.x, g4.y, ws.x, ws.y);
            dfa::fma(ut, g5.x, g5.y, wt.x, wt.y);
            F0[q] = dfa::raw(ur);
            S2[q] = dfa::raw(us);
            S3[q] = dfa::raw(ut);
        }
        __syncthreads();
        // backward: the three partials of w, into X (consumed), S4, S5
        for (int task = t; task < 3 * N2; task += T) {
            int stride;
            const int base = line_of<N>(task, stride);
            const float2 *Fd = task < N2 ? F0 : (task < 2 * N2 ? S2 : S3);
            float2 *Pd = task < N2 ? X : (task < 2 * N2 ? S4 : S5);
            line_eo<N>(Fd, Pd, base, stride, D.bwd);
        }
        if (t == 0) s_next = (long long)gridDim.x + (long long)nxt;
        __syncthreads();
        // w = sum of the partials, box faces zeroed, this thread's share of
        // <w,p>_c into its exact sum; then the next element is staged into
        // the other input array
        {
            int ex, ey, ez;
            element_coords(e, a.m, ex, ey, ez);
            const unsigned bf = box_faces(ex, ey, ez, a.m);
            const int64_t eb = e * N3;
            const double *p = a.p + eb;
            double *w = a.w + eb;
            double de = 0.0;
#pragma unroll
            for (int kk = 0; kk < PPT; kk++) {
                const int q = t + kk * T;
                if (PPT * T != N3 && q >= N3) break;
                const float2 s = dfa::add(dfa::add(X[q], S4[q]), S5[q]);
                double wv = dfa::join_scaled(s, sh_out);
                if (pf[kk] & bf)
                    wv = 0.0;
                else
                    de = fma(wv, p[q], de);
                w[q] = wv;
            }
            acc += fixed_of(de, S, a.dot_lim, out_of_range);
        }
        const int64_t en = s_next;
        if (en < a.E) stage(en, odd ? S0 : S1);
        __syncthreads();
        e = en;
    }
    return acc;
}

// CTAs per SM the register bound asks for: two or three, which hold the boxes
// that come here in one wave (df_head_elements).  As many as shared memory
// allows would spill the batched loads: 64 elements at n = 8 19.3 us per
// iteration instead of 18.2, 150 at n = 7 20.3 instead of 18.3; one CTA takes
// 31.4 us at n = 9 on 384 elements instead of 29.3.
template <int N>
__host__ __device__ constexpr int df_head_blocks() {
    constexpr int most = df_min_blocks<N, ax_df_threads(N)>(), want = N == 8 || N >= 10 ? 2 : 3;
    return most < want ? most : want;
}

template <int N>
__global__ void __launch_bounds__(ax_df_threads(N), df_head_blocks<N>())
ax_df_head_kernel(AxDfArgs a, const __grid_constant__ DfEo<N> D) {
    extern __shared__ float2 sm[];
    __shared__ double red[32];
    if (a.sc->done) return;
    const double beta = a.sc->it == 0 ? 0.0 : a.sc->beta;
    const double xa = a.sc->x_alpha;
    const double pn = a.sc->it == 0 ? a.sc->rr : a.sc->pn2;
    const int S = a.dot_shift0 - ((int)((__double_as_longlong(pn) >> 52) & 0x7ff) - 1023);
    bool out_of_range = false;
    const u128 mine = block_sum_u128(df_head_pipelined<N>(a, beta, xa, S, D, sm, out_of_range), red);
    finish_exact_sum(a.sc, a.partials, mine, S, out_of_range, a.finite && finite_pp(pn), red);
}

// ---------------------------------------------------------------- set-up
__global__ void split_scaled_kernel(const double *__restrict__ x, float2 *__restrict__ y, int64_t n,
                                    int ex) {
    const double sc = __longlong_as_double((long long)(2046 - ex) << 52);
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n;
         q += (int64_t)gridDim.x * blockDim.x)
        y[q] = dfa::split(x[q] * sc);
}

// The boxes that take this head: those whose fixed-point head would have at
// most two CTAs per SM (several elements each for n < 8 and n = 9).  A CG iteration
// with this head and with the fixed-point one, us, at 38, 152 and 304 CTAs' elements:
//   n = 2   28.1/17.9  55.2/17.9  58.2/18.8      n = 10  19.6/23.4  20.4/26.0  26.1/26.3
//   n = 4   16.5/16.8  24.0/20.6  29.9/21.9      n = 12  23.0/28.4  24.9/31.8  33.3/33.4
//   n = 6   16.1/17.8  19.7/20.6  25.3/23.9      n = 14  34.2/34.3  36.4/37.9  63.5/43.6
//   n = 8   17.1/20.8  17.7/22.8  20.3/22.1      n = 16  46.4/41.8  51.0/45.7  88.9/53.8
// So by time alone the line would lie lower at n <= 4 and at n >= 13 (where this head
// holds one CTA per SM); it lies here because the results of these boxes were kept.
bool df_head_elements(int64_t E, int n) {
    const int epc = n == 8 || n >= 10 ? 1 : (n >= 6 ? 3 : 128 / (n * n));
    return (E + epc - 1) / epc <= (int64_t)2 * device_sms();
}

// Their pairs (memory and gxyz_exp are there: prepare_fx).
nb_status prepare_df(nb_ctx *c) {
    const int64_t ng = (int64_t)6 * c->m.n * c->m.n * c->m.n * c->m.E;
    split_scaled_kernel<<<grid_blocks(ng, 256, 1024), 256, 0, c->stream>>>(c->d_gxyz, c->d_gxyz_df, ng, c->gxyz_exp);
    NB_LAUNCH_CHECK("split_scaled_kernel");
    return NB_OK;
}

// The fixed-point scale of the CG head's exact <w,p>_c: S = dot_shift0 -
// e(<p,p>_c), e the binary exponent.  Every |w_q| is at most
// A max|p| with A = 9 |D|_1 |D|_inf max|G| (three derivatives, the 3x3
// contraction, three transposed derivatives), and max|p| <= sqrt(8 <p,p>_c),
// so a thread's share of an element (P points) is below 8 P A <p,p>_c.
// sa below takes 72 P A (a further factor 9 of margin) and another 16x for
// the recursion's <p,p>_c, so the share stays below 2^(sa + e).  Summing E T shares (E elements, T threads) then
// stays below 2^(sa + e + S + log2(E T)) <= 2^125: no 128-bit sum overflows.
// The grid of the sum, 2^-S, is 2^-(125 - log2(E T)) of that bound.
template <int N>
static int dot_lim(const nb_ctx *c);

template <int N>
static int dot_shift0(const nb_ctx *c) {
    constexpr int T = ax_df_threads(N);
    constexpr int P = (N * N * N + T - 1) / T;
    double d1 = 0.0, dinf = 0.0;
    for (int i = 0; i < N; i++) {
        double rs = 0.0, cs = 0.0;
        for (int l = 0; l < N; l++) {
            rs += fabs(c->D_host[i * N + l]);
            cs += fabs(c->D_host[l * N + i]);
        }
        dinf = fmax(dinf, rs);
        d1 = fmax(d1, cs);
    }
    // max|G| < 2^(gexp - 1022)
    const int sa = (int)ceil(log2(72.0 * P * 9.0 * d1 * dinf)) + (c->gxyz_exp - 1022) + 1 + 4;
    return dot_lim<N>(c) - sa;
}

// The bound of one scaled share: 2^(125 - log2(E T)), so that E T shares
// sum below 2^125.
template <int N>
static int dot_lim(const nb_ctx *c) {
    constexpr int T = ax_df_threads(N);
    return 125 - (int)ceil(log2((double)c->m.E * T));
}

template <int N>
static nb_status launch_df_n(nb_ctx *c) {
    constexpr int T = ax_df_threads(N);
    const size_t smem = sizeof(float2) * 6 * N * N * N;
    int occ = 0;
    DfEo<N> D;
    eo_consts<N>(c->D_host, false, D.fwd);
    eo_consts<N>(c->D_host, true, D.bwd);
    AxDfArgs args{};
    args.g = c->d_gxyz_df;
    args.gexp = c->gxyz_exp;
    args.E = c->m.E;
    args.r = c->d_r;
    args.p = c->d_p;
    args.x = c->d_x;
    args.w = c->d_w;
    args.sc = c->d_sc;
    args.partials = c->d_partials;
    args.dot_shift0 = dot_shift0<N>(c) + c->test_dot_shift;
    args.dot_lim = dot_lim<N>(c);
    args.finite = c->op_finite;
    args.m = c->m;
    auto kern = ax_df_head_kernel<N>;
    {
        const nb_status s = set_smem(kern, smem);
        if (s != NB_OK) return s;
    }
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, T, smem);
    if (occ < 1) occ = 1;
    const int64_t cap = (int64_t)device_sms() * occ;
    const int grid = (int)(c->m.E < cap ? c->m.E : cap);
    c->ax_grid = grid;
    LaunchTimer tm(c, NB_K_AX);
    kern<<<grid, T, smem, c->stream>>>(args, D);
    NB_LAUNCH_CHECK("ax_df_head_kernel");
    return NB_OK;
}

nb_status launch_df_head(nb_ctx *c) {
    switch (c->m.n) {
#define NB_CASE(NN) case NN: return launch_df_n<NN>(c);
        NB_CASE(2) NB_CASE(3) NB_CASE(4) NB_CASE(5) NB_CASE(6) NB_CASE(7) NB_CASE(8)
        NB_CASE(9) NB_CASE(10) NB_CASE(11) NB_CASE(12) NB_CASE(13) NB_CASE(14) NB_CASE(15)
        NB_CASE(16)
#undef NB_CASE
    }
    return fail(NB_ERR_ARG, "unsupported n");
}

}  // namespace nekgb
