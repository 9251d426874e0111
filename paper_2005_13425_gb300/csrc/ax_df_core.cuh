// Double-float ax_e (Listing 1, arXiv 2005.13425 Sec. III) on FP32 pairs
// (df.cuh) for the batched engine (engine.cu), the CG head on boxes of few
// elements (ax_df.cu), the fixed-point kernels' graded elements
// (ax_fx_core.cuh) and the measurement probe (probe_tc.cu): derivative-matrix
// constants, the line products and one element of the operator.
#pragma once

#include "df.cuh"
#include "internal.cuh"
#include "reduce.cuh"

namespace nekgb {

// Even-odd form of a centro-antisymmetric matrix M (M(N-1-m, N-1-l) =
// -M(m,l), which holds for the GLL derivative matrix and its transpose).
// With H = N/2, xs_l = x_l + x_{N-1-l}, xd_l = x_l - x_{N-1-l} (l < H):
//   y_m       = P_m + Q_m,   y_{N-1-m} = P_m - Q_m   (m < H)
//   P_m = sum_{l<H} a(m,l) xd_l,            a(m,l) = (M(m,l) + M(N-1-m,l))/2
//   Q_m = sum_{l<H} b(m,l) xs_l + b(m,H) x_H, b(m,l) = (M(m,l) - M(N-1-m,l))/2
// and for odd N the middle output y_H = sum_{l<H} M(H,l) xd_l + M(H,H) x_H.
// This halves the products of a line (Solomonoff's even-odd decomposition).
// The outputs are stored as unnormalised pairs (dfa::add_acc_raw).
template <int N>
struct EoMat {
    static constexpr int H = N / 2;
    float ah[H * H], al[H * H];
    float bh[H * (H + 1)], bl[H * (H + 1)];
    float ch[H + 1], cl[H + 1];
};

template <int N>
struct DfEo {
    EoMat<N> fwd;   // M = D
    EoMat<N> bwd;   // M = D^T
};

// The plain form, for a matrix that is not centro-antisymmetric.
template <int N>
struct DfMat {
    struct Half {
        float h[N * N], l[N * N];
    } fwd, bwd;
};

template <int N, bool EO>
struct DfConsts;
template <int N>
struct DfConsts<N, false> { using type = DfMat<N>; };
template <int N>
struct DfConsts<N, true> { using type = DfEo<N>; };


// One line task per thread up to n = 12; two per thread above, so that the
// n-long line held in registers does not spill at n = 16.
__host__ __device__ constexpr int ax_df_threads(int n) {
    return n <= 12 ? ((3 * n * n + 31) / 32) * 32 : ((3 * n * n + 1) / 2 + 31) / 32 * 32;
}

// Threads of a CTA that gives each thread `lpt` line tasks (lpt >= 1).
__host__ __device__ constexpr int df_threads_lpt(int n, int lpt) {
    return ((3 * n * n + lpt - 1) / lpt + 31) / 32 * 32;
}

// CTAs of T threads per SM that the register bound of a kernel around the
// element operator asks for: as many as the six n^3 pair arrays allow in
// 228 KB of shared memory (1 KB reserved per CTA), but no more than leave R
// registers per thread (a line at n <= 10 needs 48; the batched kernel's
// tile head then spills about 100 bytes at n = 10, which costs less than
// the CTA a 64-register bound loses); 4 at n = 10, 2 at n = 11, 12 for R = 48.
// Above n = 12 a line's registers cannot be bounded without spilling.
template <int N, int T, int R = 48>
__host__ __device__ constexpr int df_min_blocks() {
    constexpr int by_smem = (228 * 1024) / (6 * N * N * N * 8 + 1024);
    constexpr int by_regs = 65536 / (T * R);
    return N > 12 ? 1 : (N > 10 ? by_smem : (by_smem < by_regs ? by_smem : by_regs));
}

// Line task -> (first point, stride) of the line and the direction.
template <int N>
__device__ __forceinline__ int line_of(int task, int &stride) {
    constexpr int N2 = N * N;
    const int d = task / N2;
    const int c = task - d * N2;
    const int a0 = c % N, a1 = c / N;
    if (d == 0) {        // along r: line (j = a0, k = a1)
        stride = 1;
        return N * (a0 + N * a1);
    }
    if (d == 1) {        // along s: line (i = a0, k = a1)
        stride = N;
        return a0 + N2 * a1;
    }
    stride = N2;         // along t: line (i = a0, j = a1)
    return a0 + N * a1;
}

// out(base + m*stride) = sum_l M(m,l) in(base + l*stride) in even-odd form
// (see EoMat): pair sums and differences, then 2 dot products of N/2 terms per
// output pair.
template <int N>
__device__ __forceinline__ void line_eo(const float2 *in, float2 *out, int base, int stride,
                                        const EoMat<N> &M) {
    constexpr int H = N / 2;
    float sh[H], sl[H], dh[H], dl[H];
#pragma unroll
    for (int l = 0; l < H; l++) {
        const float2 a = in[base + l * stride], b = in[base + (N - 1 - l) * stride];
        const float2 s = dfa::add(a, b);
        const float2 d = dfa::add(a, make_float2(-b.x, -b.y));
        sh[l] = s.x; sl[l] = s.y;
        dh[l] = d.x; dl[l] = d.y;
    }
    float ch = 0.f, cl = 0.f;
    if (N & 1) {
        const float2 c = in[base + H * stride];
        ch = c.x;
        cl = c.y;
    }
#pragma unroll
    for (int m = 0; m < H; m++) {
        dfa::Acc P = dfa::first(M.ah[m * H], M.al[m * H], dh[0], dl[0]);
#pragma unroll
        for (int l = 1; l < H; l++) dfa::fma(P, M.ah[m * H + l], M.al[m * H + l], dh[l], dl[l]);
        dfa::Acc Q = dfa::first(M.bh[m * (H + 1)], M.bl[m * (H + 1)], sh[0], sl[0]);
#pragma unroll
        for (int l = 1; l < H; l++) dfa::fma(Q, M.bh[m * (H + 1) + l], M.bl[m * (H + 1) + l], sh[l], sl[l]);
        if (N & 1) dfa::fma(Q, M.bh[m * (H + 1) + H], M.bl[m * (H + 1) + H], ch, cl);
        out[base + m * stride] = dfa::add_acc_raw(P, Q, 1.f);
        out[base + (N - 1 - m) * stride] = dfa::add_acc_raw(P, Q, -1.f);
    }
    if (N & 1) {
        dfa::Acc Y = dfa::first(M.ch[0], M.cl[0], dh[0], dl[0]);
#pragma unroll
        for (int l = 1; l < H; l++) dfa::fma(Y, M.ch[l], M.cl[l], dh[l], dl[l]);
        dfa::fma(Y, M.ch[H], M.cl[H], ch, cl);
        out[base + H * stride] = dfa::norm(Y);
    }
}

// The same in plain form, the outputs as unnormalised pairs.
template <int N>
__device__ __forceinline__ void line_plain(const float2 *in, float2 *out, int base, int stride,
                                           const typename DfMat<N>::Half &M) {
    float2 x[N];
#pragma unroll
    for (int l = 0; l < N; l++) x[l] = in[base + l * stride];
#pragma unroll 1
    for (int m = 0; m < N; m++) {
        dfa::Acc acc = dfa::first(M.h[m * N], M.l[m * N], x[0].x, x[0].y);
#pragma unroll
        for (int l = 1; l < N; l++) dfa::fma(acc, M.h[m * N + l], M.l[m * N + l], x[l].x, x[l].y);
        out[base + m * stride] = dfa::raw(acc);
    }
}

// u = g w at one point, in place: g = (rr, rs, rt, ss, st, tt).
__device__ __forceinline__ void df_contract(const float2 (&g)[6], float2 &a, float2 &b, float2 &c) {
    auto row = [&](int q0, int q1, int q2) {
        dfa::Acc u = dfa::first(g[q0].x, g[q0].y, a.x, a.y);
        dfa::fma(u, g[q1].x, g[q1].y, b.x, b.y);
        dfa::fma(u, g[q2].x, g[q2].y, c.x, c.y);
        return dfa::raw(u);
    };
    const float2 r = row(0, 1, 2), s = row(1, 3, 4), t = row(2, 4, 5);
    a = r;
    b = s;
    c = t;
}

// Points of an element per thread of a T-thread CTA in the pointwise phases.
template <int N, int T>
__host__ __device__ constexpr int df_points_per_thread() {
    return (N * N * N + T - 1) / T;
}

// w = ax_e(u) on one element in double-float arithmetic, executed by the whole
// CTA (every thread must call it; it contains barriers).  u, w: the element's
// points, g: its gxyz pairs [6][n^3], unscaled.  sm holds 6 n^3 pairs, s_emax
// is a shared int that must be 0 on entry (left 0 on exit).
template <int N, int T>
__device__ __forceinline__ void df_element(const double *u, double *w, const float2 *g, const DfEo<N> &D, float2 *sm,
                                           int *s_emax) {
    constexpr int N2 = N * N, N3 = N * N * N;
    float2 *U = sm;            // input pairs; later the r-partial of w
    float2 *W0 = sm + N3;      // wr -> ur
    float2 *W1 = sm + 2 * N3;  // ws -> us
    float2 *W2 = sm + 3 * N3;  // wt -> ut
    float2 *P1 = sm + 4 * N3;  // s-partial of w
    float2 *P2 = sm + 5 * N3;  // t-partial of w
    double *raw = reinterpret_cast<double *>(U);
    const int t = threadIdx.x;
    // ---- stage the element (raw FP64 first, to find its scale)
    int emax = 0;
    for (int q = t; q < N3; q += T) {
        const double v = __ldg(u + q);
        raw[q] = v;
        const int exb = (int)((__double_as_longlong(v) >> 52) & 0x7ff);
        emax = exb > emax ? exb : emax;
    }
    emax = __reduce_max_sync(0xffffffffu, emax);
    if ((t & 31) == 0) atomicMax(s_emax, emax);
    __syncthreads();
    int eu = *s_emax;
    eu = eu < 1 ? 1 : (eu > 2046 ? 2046 : eu);
    // u is scaled by 2^(1023-eu) so the element's max is in [1,2); w is
    // scaled back by 2^(eu-1023)
    const int sh_in = 1023 - eu, sh_out = eu - 1023;
    for (int q = t; q < N3; q += T) U[q] = dfa::split_scaled(raw[q], sh_in);  // own entries only
    __syncthreads();

    // ---- forward: wr, ws, wt along this thread's line
    for (int task = t; task < 3 * N2; task += T) {
        int stride;
        const int base = line_of<N>(task, stride);
        line_eo<N>(U, task < N2 ? W0 : (task < 2 * N2 ? W1 : W2), base, stride, D.fwd);
    }
    __syncthreads();

    // ---- geometric contraction, pointwise, in place
    for (int q = t; q < N3; q += T) {
        const float2 wr = W0[q], ws = W1[q], wt = W2[q];
        const float2 g0 = __ldcs(g + q), g1 = __ldcs(g + N3 + q), g2 = __ldcs(g + 2 * N3 + q);
        const float2 g3 = __ldcs(g + 3 * N3 + q), g4 = __ldcs(g + 4 * N3 + q), g5 = __ldcs(g + 5 * N3 + q);
        dfa::Acc r = dfa::first(g0.x, g0.y, wr.x, wr.y);
        dfa::fma(r, g1.x, g1.y, ws.x, ws.y);
        dfa::fma(r, g2.x, g2.y, wt.x, wt.y);
        dfa::Acc s = dfa::first(g1.x, g1.y, wr.x, wr.y);
        dfa::fma(s, g3.x, g3.y, ws.x, ws.y);
        dfa::fma(s, g4.x, g4.y, wt.x, wt.y);
        dfa::Acc tt = dfa::first(g2.x, g2.y, wr.x, wr.y);
        dfa::fma(tt, g4.x, g4.y, ws.x, ws.y);
        dfa::fma(tt, g5.x, g5.y, wt.x, wt.y);
        W0[q] = dfa::raw(r);
        W1[q] = dfa::raw(s);
        W2[q] = dfa::raw(tt);
    }
    __syncthreads();

    // ---- backward: w_d(m) = sum_l dxtm1(m,l) u_d(l) = sum_l D(l,m) u_d(l)
    for (int task = t; task < 3 * N2; task += T) {
        int stride;
        const int base = line_of<N>(task, stride);
        line_eo<N>(task < N2 ? W0 : (task < 2 * N2 ? W1 : W2), task < N2 ? U : (task < 2 * N2 ? P1 : P2), base,
                   stride, D.bwd);
    }
    __syncthreads();

    // ---- w = r-partial + s-partial + t-partial, scaled back, FP64 out
    for (int q = t; q < N3; q += T)
        w[q] = dfa::join_scaled(dfa::add(dfa::add(U[q], P1[q]), P2[q]), sh_out);
    if (t == 0) *s_emax = 0;
    __syncthreads();
}

// Even-odd constants of M (M = D, or D^T when tr) from the FP64 matrix.
template <int N>
inline void eo_consts(const double *Dm, bool tr, EoMat<N> &E) {
    constexpr int H = N / 2;
    auto M = [&](int mm, int l) { return tr ? Dm[l * N + mm] : Dm[mm * N + l]; };
    auto put = [](double v, float &h, float &l) {
        h = (float)v;
        l = (float)(v - (double)h);
    };
    for (int mm = 0; mm < H; mm++) {
        for (int l = 0; l < H; l++) put(0.5 * (M(mm, l) + M(N - 1 - mm, l)), E.ah[mm * H + l], E.al[mm * H + l]);
        for (int l = 0; l <= H; l++) {
            const double v = l < H ? 0.5 * (M(mm, l) - M(N - 1 - mm, l)) : ((N & 1) ? M(mm, H) : 0.0);
            put(v, E.bh[mm * (H + 1) + l], E.bl[mm * (H + 1) + l]);
        }
    }
    for (int l = 0; l <= H; l++) put((N & 1) ? M(H, l) : 0.0, E.ch[l], E.cl[l]);
}

template <int N, bool EO>
inline void df_consts(const double *Dm, typename DfConsts<N, EO>::type &C) {
    if constexpr (EO) {
        eo_consts<N>(Dm, false, C.fwd);
        eo_consts<N>(Dm, true, C.bwd);
    } else {
        auto put = [](double v, float &h, float &l) {
            h = (float)v;
            l = (float)(v - (double)h);
        };
        for (int m = 0; m < N; m++)
            for (int l = 0; l < N; l++) {
                put(Dm[m * N + l], C.fwd.h[m * N + l], C.fwd.l[m * N + l]);
                put(Dm[l * N + m], C.bwd.h[m * N + l], C.bwd.l[m * N + l]);
            }
    }
}

}  // namespace nekgb
