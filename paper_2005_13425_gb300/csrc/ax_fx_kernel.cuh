// ax_e in fixed-point pairs: the element-local Poisson operator of Listing 1
// (arXiv 2005.13425, Sec. III) to FP64 accuracy on GB300's integer and FP32
// pipes (its FP64 pipe delivers only ~1 TFLOP/s).
//
// Arithmetic.  u, gxyz and D are pairs of a 32-bit integer and a float
// (fx.cuh): the leading products are summed exactly in 64-bit integers, the
// small ones in FP32.  Inputs are scaled by exact powers of two (per element
// for u and gxyz), so the data's magnitude does not matter; the output is
// scaled back exactly and rounded once.
//
// Thread layout.  A thread owns a column of an element along t and a line along
// r and s (ax_fx_core.cuh): the t derivatives and the contraction with the
// six geometric factors (streamed from HBM, coalesced) stay in its registers,
// the r and s values pass through shared memory.  The entries of D are
// compile-time indexed kernel parameters, so they are constant operands and
// cost no loads.  Five barriers per element.
#pragma once

#include <math.h>

#include <type_traits>

#include "ax_fx_core.cuh"
#include "exact_sum.cuh"

namespace nekgb {

struct AxFxArgs {
    const double *u;      // MODE 0 input
    double *w;            // output (FP64, local storage)
    const double *r;      // MODE 1, 2: residual
    double *p;            // MODE 1, 2: search direction, updated in place
    double *x;            // MODE 1, 2: iterate, receives the owed x += x_alpha p
    const double *minv;   // MODE 1: Jacobi inverse diagonal or null
    CgScalars *sc;        // MODE 1, 2
    double *partials;     // MODE 1 with fuse, MODE 2: one <w,p> partial per CTA
    int dot_shift0;       // MODE 2: scale of the exact <w,p>_c sum (see launch_fx_nv)
    int dot_lim;          // MODE 2: a share of 2^dot_lim or more (scaled) may overflow the sum
    int finite;           // MODE 2: the operator's data (D and gxyz) has no NaN or Inf
    int fuse;             // MODE 1: zero box-face points, local products w p
    Mesh m;
    FxData fd;
    int64_t E;
};

// v 2^k truncated to an integer, as a two's-complement 128-bit value.  The
// caller's k keeps |v| 2^k below 2^lim (lim = 125 - log2 of the number of
// shares, see the head), so no sum of shares overflows; a share that may
// reach 2^lim sets `out_of_range` (the solve then stops with a status instead
// of using a wrong sum).
__device__ __forceinline__ u128 fixed_of(long long v, int k, int lim, bool &out_of_range) {
    if (v == 0) return 0;
    out_of_range |= 64 - __clzll(v < 0 ? -v : v) + k > lim;
    if (k < 0) return k > -64 ? (u128)(__int128)(v >> -k) : (u128)0;
    return (u128)(__int128)v << (k < 127 ? k : 127);
}

// The unpreconditioned two-kernel CG head with a software-pipelined,
// dynamically scheduled element loop.
//
// Scale.  An element's pairs of p are scaled by its largest exponent, a
// maximum over the CTA (one warp reduction and one shared atomic per warp, and
// one barrier).  A scale for the whole iteration, from <p,p>_c, needs no
// reduction but lies up to sqrt(8 N) above the largest entry (2^13 on the
// largest box), which a fixed-point pair does not have to spare.
//
// Pipeline.  The next elements' p is formed in registers while the final pass
// reads the current partials, and goes into X after one barrier, when its
// largest exponent is known.
//
// Schedule.  After its first elements (blockIdx.x) a CTA takes the next ones
// from a counter in the scalar block, so SMs that run slower take fewer
// (a static assignment left the slowest SM 12 % behind the mean).  The
// counter is read at the start of a step and published just before the
// barrier that ends the backward pass, which hides the atomic's latency.
// <w,p>_c stays independent of the schedule because it is summed exactly:
// each thread's share of an element (its points' products of the fixed-point
// pairs of w and p, an integer) is shifted to the fixed scale 2^S (fixed_of,
// truncating) and added to the thread's 128-bit integer sum; integer sums do
// not depend on the order of the additions.  The caller chooses S from
// <p,p>_c and a bound on the operator so that no sum can overflow (see
// launch_fx_nv); the result is rounded to FP64 once, at the end.
template <int N, bool EO, int G>
__device__ __forceinline__ u128 cg_head_pipelined(const AxFxArgs &a, double beta, double xa, int S128,
                                                  const typename FxConsts<N, EO>::type &D, int2 *sm,
                                                  unsigned *s_max, FxList<fx_epc(N, G), true> &list,
                                                  bool &out_of_range) {
    constexpr int N3 = N * N * N, A = fx_array(N), EPC = fx_epc(N, G);
    constexpr bool KEEP = fx_keep(N, G);
    __shared__ long long s_next;
    FxThread<N, G> th;
    th.init();
    int2 *X = sm + (KEEP ? 4 : 3) * A * th.el, *R = X + A, *S = X + 2 * A, *TT = KEEP ? X + 3 * A : X;
    const int col = th.column();
    double v[FxThread<N, G>::K];
    unsigned top = 0;
    auto load = [&](int64_t e0) {   // the direction, kept in v
        const int64_t e = e0 + th.el, q = e * N3 + col;
        const bool on = th.active && e < a.E;
        if (on) {
            fx_direction<N, false>(th, a.r + q, a.p + q, a.x + q, nullptr, beta, xa, v);
            top = fx_top_of(th, v);
        }
        fx_max_in(th, on, top, s_max);
    };
    u128 acc = 0;
    int64_t e0 = (int64_t)blockIdx.x * EPC;
    if (e0 < a.E) load(e0);
    __syncthreads();
    while (e0 < a.E) {
        const int64_t e = e0 + th.el;
        const bool on = th.active && e < a.E;
        unsigned nxt = 0;
        if (threadIdx.x == 0) nxt = atomicAdd(&a.sc->next_elem, 1u);
        const unsigned elem = s_max[th.el];
        const int emax = fx_emax(elem);
        if (EPC > 1) fx_mark_small(th, a.fd, on, top, elem, s_max);
        if (on) fx_put_input(th, v, emax, X);
        __syncthreads();
        if (threadIdx.x < EPC) {
            const unsigned etop = s_max[threadIdx.x];
            s_max[threadIdx.x] = 0;
            fx_note<N, G>(a.fd, e0, a.E, etop, s_max + EPC, list);
        }
        fx_operator<N, EO>(th, on, X, R, S, TT, a.fd.g + e * 3 * N3 + col, D, s_max + EPC);
        if (threadIdx.x == 0) s_next = ((long long)gridDim.x + (long long)nxt) * EPC;
        __syncthreads();
        if (on) {   // w, and this thread's share of <w,p>_c into its exact sum
            int ex, ey, ez;
            element_coords(e, a.m, ex, ey, ez);
            const int so = emax + (a.fd.ge[e] & kFxExp) + D.so0;
            fx_final(th, X, R, S, TT, a.w + e * N3 + col, a.p + e * N3 + col, so, emax, box_faces(ex, ey, ez, a.m),
                     [&](long long dA, float dB) {
                         acc += fixed_of(dA + __float2ll_rn(dB), S128 + so + emax - 1052, a.dot_lim, out_of_range);
                     });
        }
        const int64_t en = s_next;
        if (en < a.E) load(en);
        __syncthreads();
        e0 = en;
    }
    return acc;
}

// MODE 0: w = ax_e(u); 1: the CG head of the forms with further kernels
// (Jacobi, mask array); 2: the two-kernel CG's head.  As many CTAs per SM as
// registers and shared memory hold (fx_min_blocks).
template <int N, int MODE, bool EO, int G>
__global__ void __launch_bounds__(fx_threads(N, G), fx_min_blocks<N, G, MODE == 2 && fx_keep(N, G)>())
ax_fx_kernel(const __grid_constant__ AxFxArgs a, const __grid_constant__ typename FxConsts<N, EO>::type D) {
    constexpr int EPC = fx_epc(N, G);
    extern __shared__ __align__(16) int2 sm[];
    __shared__ unsigned s_max[2 * EPC];
    __shared__ FxList<EPC, MODE != 0> list;
    __shared__ double red[32];
    double beta = 0.0, xa = 0.0, dot = 0.0;
    if (MODE != 0) {
        if (a.sc->done) return;
        beta = a.sc->it == 0 ? 0.0 : a.sc->beta;
        xa = a.sc->x_alpha;
    }
    if (threadIdx.x < EPC) s_max[threadIdx.x] = s_max[EPC + threadIdx.x] = 0;
    list.init();
    __syncthreads();
    if constexpr (MODE == 2) {
        // the exact sums: per CTA, then over the CTAs by the last one
        const double pn = a.sc->it == 0 ? a.sc->rr : a.sc->pn2;
        const int S = a.dot_shift0 - ((int)((__double_as_longlong(pn) >> 52) & 0x7ff) - 1023);
        bool out_of_range = false;
        const u128 mine = block_sum_u128(cg_head_pipelined<N, EO, G>(a, beta, xa, S, D, sm, s_max, list, out_of_range), red);
        if (list.head >= 0) fx_redo_list<N, EO, G>(a.fd, list, a.p, a.w, true, a.m, sm, fx_keep(N, G) ? 4 : 3);
        finish_exact_sum(a.sc, a.partials, mine, S, out_of_range, a.finite && finite_pp(pn), red);
    } else {
        FxThread<N, G> th;
        th.init();
        FxIO io;
        io.u = a.u;
        io.r = a.r;
        io.p = a.p;
        io.x = a.x;
        io.minv = a.minv;
        io.w = a.w;
        for (int64_t e0 = (int64_t)blockIdx.x * EPC; e0 < a.E; e0 += (int64_t)gridDim.x * EPC)
            fx_elements<N, MODE, EO, G>(io, a.fd, e0, a.E, beta, xa, a.fuse != 0, a.m, th, D, sm, s_max,
                                        list, dot);
        if (list.head >= 0)
            fx_redo_list<N, EO, G>(a.fd, list, MODE == 0 ? a.u : a.p, a.w, MODE == 1 && a.fuse, a.m, sm,
                                   G == 3 ? 4 : 3);
        if (MODE == 1 && a.fuse) {
            const double b = block_sum(dot, red);
            if (threadIdx.x == 0) a.partials[blockIdx.x] = b;
        }
    }
}

template <int N, bool EO, int G>
static nb_status launch_fx_nv(nb_ctx *c, const double *u, double *w, int mode) {
    constexpr int T = fx_threads(N, G), EPC = fx_epc(N, G);
    // the two-kernel CG (box mask, no preconditioner) has its own head
    const bool head = mode == 1 && c->two_kernel;
    const size_t smem = fx_smem_bytes(N, G, head && fx_keep(N, G));
    int occ = 0;
    const auto &D = *reinterpret_cast<const typename FxConsts<N, EO>::type *>(c->fx_tab.data());
    AxFxArgs args{};
    args.fd = {c->d_gxyz_fx, c->d_ge, c->d_gxyz, c->d_D_df, c->gxyz_exp, c->fx_special,
               c->d_redo_list};
    args.E = c->m.E;
    if (mode == 0) {
        args.u = u;
        args.w = w;
    } else {
        args.r = c->d_r;
        args.p = c->d_p;
        args.x = c->d_x;
        args.minv = c->d_minv;
        args.w = c->d_w;
        args.sc = c->d_sc;
        args.partials = c->d_partials;
        args.fuse = c->fused_cg ? 1 : 0;
        args.dot_shift0 = c->fx_dot_shift0 + c->test_dot_shift;
        args.dot_lim = c->fx_dot_lim;
        args.finite = c->op_finite;
    }
    args.m = c->m;
    auto kern = mode == 0 ? ax_fx_kernel<N, 0, EO, G> : ax_fx_kernel<N, 1, EO, G>;
    if constexpr (G == 1) {
        static_assert(2 * (T / 32) <= 32, "block_sum_u128's scratch");
        if (head) kern = ax_fx_kernel<N, 2, EO, G>;
    }
    {
        const nb_status s = set_smem(kern, smem);
        if (s != NB_OK) return s;
    }
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, T, smem);
    if (occ < 1) occ = 1;
    const int64_t cap = (int64_t)device_sms() * occ, need = (c->m.E + EPC - 1) / EPC;
    // the operator alone: one CTA per group of elements, which the hardware
    // hands out as SMs become free (a resident grid striding over 4096 elements
    // at n = 10 idled a tenth of the time in its last round; FxList relies on one
    // group); the heads: a resident grid, one reduction per CTA
    const int64_t most = mode == 0 ? (int64_t)0x7fffffff : cap;
    const int grid = (int)(need < most ? need : most);
    if (mode == 1) c->ax_grid = grid;
    LaunchTimer tm(c, NB_K_AX);
    kern<<<grid, T, smem, c->stream>>>(args, D);
    NB_LAUNCH_CHECK("ax_fx_kernel");
    return NB_OK;
}

// The tables of a context (c->fx_tab), made once: they take the host 5 to 20 us.
template <int N>
void fx_tables_n(nb_ctx *c) {
    auto make = [&](auto *D, auto eo) {
        using T = std::remove_pointer_t<decltype(D)>;
        static_assert(sizeof(T) % sizeof(int4) == 0, "");
        c->fx_tab.resize(sizeof(T) / sizeof(int4));
        constexpr bool EO = decltype(eo)::value;
        using Df = typename DfConsts<N, EO>::type;
        static_assert(sizeof(Df) <= sizeof(float) * fx_df_floats(N), "");
        c->df_tab.resize(sizeof(Df) / sizeof(float));
        for (int q = 0; q < N * N; q++)
            if (!isfinite(c->D_host[q])) return;   // see prepare_fx
        fx_consts<N, EO>(c->D_host, *reinterpret_cast<T *>(c->fx_tab.data()));
        df_consts<N, EO>(c->D_host, *reinterpret_cast<Df *>(c->df_tab.data()));
    };
    if (c->d_eo) make((typename FxConsts<N, true>::type *)nullptr, std::true_type{});
    else make((typename FxConsts<N, false>::type *)nullptr, std::false_type{});
}

template <int N>
nb_status launch_fx_n(nb_ctx *c, const double *u, double *w, int mode) {
    if (!c->d_eo) return launch_fx_nv<N, false, 1>(c, u, w, mode);
    const bool head = mode == 1 && c->two_kernel;   // on few elements: ax_df.cu
    if (fx_few_elements(c->m.E, N) && !head) return launch_fx_nv<N, true, 3>(c, u, w, mode);
    return launch_fx_nv<N, true, 1>(c, u, w, mode);
}

}  // namespace nekgb
