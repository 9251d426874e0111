// Core of the FP64-accurate ax_e (Listing 1, arXiv 2005.13425 Sec. III) in
// fixed-point pairs (fx.cuh) for the kernels of ax_fx_kernel.cuh: the scaled
// derivative-matrix constants, the line products (plain and even-odd), the
// phases of one element, the elements that are computed again in double-float
// arithmetic, and the conversion of the geometric factors.
//
// Scales.
//  * The rows of D are brought to similar size and the geometric factors take
//    the difference: with D^ = diag(c) D and g^_de = g_de rho(d) rho(e), rho the
//    reciprocal of c at the point's index along d, D^^T g^ D^ = D^T g D.
//    c(m) is the row's absolute sum to the power -3/4.  (At n = 10 the end rows
//    of D are six times the middle ones, and the quadrature weights in g run
//    the other way; without this the error is 4 to 30 times larger, with the
//    power 1 or 1/2 twice.)
//  * D^ is multiplied by kf (forward) and kb (transposed) so that the absolute
//    sums of its rows are at most 2^32 and its entries below 2^31; rho takes
//    1/sqrt(mu) of kf kb = 2^k mu, so that only a power of two remains.
//    g^ is rounded to 53 bits once more, D^ to 55: everything else is exact.
//  * An element of the input has its largest exponent emax: |h| < 2^30.
//  * The six factors of a point share a scale (exponent eq) with which the
//    largest absolute row sum of the 3 x 3 matrix lies in (2^30, 2^31]; the
//    element has ge = max eq, and the shift s = ge - eq (at most 31) stands
//    in the low 5 bits of the rr factor's float, where it costs that factor
//    2^-50 of its size.
// Then |h| < 2^30 after the forward products, 2^29 after the contraction and
// 2^29 in each of the three partials, and the operator's result is
// (h + l) 2^so with so = emax + ge - k - 2009.
#pragma once

#include "ax_df_core.cuh"
#include "fx.cuh"
#include "internal.cuh"
#include "reduce.cuh"

namespace nekgb {

// Scaled constants, 16 bytes each (one uniform load): h = rint(v k), l the rest
// and f = (float)h, both times 2^-32.
struct __align__(16) FxConst {
    int h;
    float l, f;
    int pad;
};
template <int M>
struct FxTab {
    FxConst v[M];
};

// A copy of the tables per direction: the line bodies of the three directions
// would otherwise read the same constants, and the compiler keeps what it has
// read once in spilled registers (6.4 KB a thread at n = 16).
template <int N>
struct FxMat {
    FxTab<N * N> fwd[3];   // D^ kf, entry m*N + l
    FxTab<N * N> bwd[3];   // D^^T kb
    int so0, pad[3];    // -k - 2009
};

// Even-odd form of a centro-antisymmetric matrix M (M(N-1-m, N-1-l) =
// -M(m,l), which holds for the GLL derivative matrix and its transpose).
// With H = N/2, xs_l = x_l + x_{N-1-l}, xd_l = x_l - x_{N-1-l} (l < H):
//   y_m       = P_m + Q_m,   y_{N-1-m} = P_m - Q_m   (m < H)
//   P_m = sum_{l<H} a(m,l) xd_l,            a(m,l) = (M(m,l) + M(N-1-m,l))/2
//   Q_m = sum_{l<H} b(m,l) xs_l + b(m,H) x_H, b(m,l) = (M(m,l) - M(N-1-m,l))/2
// and for odd N the middle output y_H = sum_{l<H} M(H,l) xd_l + M(H,H) x_H.
// This halves the products of a line (Solomonoff's even-odd decomposition).
// b(m,H) stands after the H x H part, at H*H + m.
template <int N>
struct FxEoHalf {
    static constexpr int H = N / 2;
    FxTab<H * H> a;
    FxTab<H * H + H> b;
    FxTab<H + 1> c;
};
template <int N>
struct FxEo {
    FxEoHalf<N> fwd[3], bwd[3];
    int so0, pad[3];
};

template <int N, bool EO>
struct FxConsts;
template <int N>
struct FxConsts<N, false> { using type = FxMat<N>; };
template <int N>
struct FxConsts<N, true> { using type = FxEo<N>; };

// Thread layout, G = 1 (throughput).  Thread (i, j) of an element owns its
// column along t (points (i, j, 0..n-1)) in every pointwise step, the t line
// there, one line along r (j' = j, k' = i) and one along s (i' = i, k' = j).  So
// the t lines and the contraction need no exchange between threads, and a CTA
// is small: five per SM at n = 10, in different phases.  (With one line of any
// direction per thread a CTA has three times the threads, two or three fit an
// SM and their phases meet: 4096 elements at n = 10 took 93 us instead of 86,
// 504 at n = 16 113 instead of 60.)  Small orders put several elements into one CTA.
// G = 3 (latency, for fewer elements than keep the SMs busy): three threads per
// column, of which thread d owns the line along direction d and every third
// point of the column; a barrier more.
__host__ __device__ constexpr int fx_epc(int n, int G) {   // elements per CTA
    return G == 3 || n == 8 || n >= 10 ? 1 : (n >= 6 ? 3 : 128 / (n * n));
}
__host__ __device__ constexpr int fx_threads(int n, int G) { return (fx_epc(n, G) * G * n * n + 31) / 32 * 32; }

// Few elements: at most two CTAs per SM in the throughput layout (one element
// each; n = 6 and 7 put three into a CTA).  64 elements at n = 8 take 6.2 us with
// three threads per column and 8.2 with one; 384 elements 8.2 at n = 7 and 8
// either way, at n = 9 14.4 and 10.3; 4096 at n = 8 52 and 38.  At
// n = 4 64 elements take 4.6 and 6.1 us, 384 6.2 and 6.1.
inline bool fx_few_elements(int64_t E, int n) {
    return E <= (int64_t)2 * device_sms() * (n == 6 || n == 7 ? 3 : 1);
}

// Layout of an element's pairs in shared memory: point (i, j, k) at i + n j +
// L k.  15 of a point's 23 accesses (8 bytes each) go along a column, whose
// neighbours are consecutive: no bank conflicts.  With L odd, the lines along
// r of 16 neighbouring threads (thread (i, j) takes the line (j, k = i))
// start in 16 different bank pairs as well; those along s are two-way.
__host__ __device__ constexpr int fx_layer(int n) { return n * n + (n % 2 ? 0 : (n % 4 ? 5 : 1)); }
__host__ __device__ constexpr int fx_array(int n) { return fx_layer(n) * n; }

// Arrays per element: the input, the r, s and t values; without `keep` (G = 1
// only) the t values take the input's place.
__host__ __device__ constexpr size_t fx_smem_bytes(int n, int G, bool keep) {
    return sizeof(int2) * (keep || G == 3 ? 4 : 3) * fx_array(n) * fx_epc(n, G);
}
// The CG heads keep the input for the products w p up to n = 12; above, where
// a fourth array would cost a CTA, they form it again from p.
__host__ __device__ constexpr bool fx_keep(int n, int G) { return n <= 12 || G == 3; }

// CTAs per SM that the register bound of a kernel around the element operator
// asks for: as many as leave 96 registers per thread (128 above n = 12, where
// a line is longer) and as the shared memory holds (228 KB, 1 KB reserved per
// CTA).  At 80 registers the heads spill and are 10 % slower, one CTA more or
// not.
template <int N, int G, bool KEEP>
__host__ __device__ constexpr int fx_min_blocks() {
    constexpr int by_smem = (228 * 1024) / ((int)fx_smem_bytes(N, G, KEEP) + 1024);
    constexpr int by_regs = 65536 / (fx_threads(N, G) * (N > 12 && G == 1 ? 128 : 96));
    constexpr int b = by_smem < by_regs ? by_smem : by_regs;
    return b < 1 ? 1 : (b > 24 ? 24 : b);
}

// Exponents below the element's largest from which entries count as small (see
// Graded elements).
__host__ __device__ constexpr int fx_grade(int n) { return n <= 3 ? 10 : 8; }
// Top words of elements that are graded because all their entries are tiny.
constexpr unsigned kFxTiny = (unsigned)(fx::kMinExp + 1) << 20;

// A thread's place: its element within the CTA's group, (i, j) and, with
// G = 3, its number d in the column.
template <int N, int G>
struct FxThread {
    static constexpr int K = (N + G - 1) / G;   // points of the column per thread: k = d, d + G, ...
    int el, i, j, d;
    bool active;       // the thread has a column
    __device__ __forceinline__ void init() {
        constexpr int N2 = N * N, EPC = fx_epc(N, G);
        const int t = threadIdx.x;
        d = G == 1 ? 0 : t / N2;
        const int u = t - d * N2;
        el = EPC == 1 ? 0 : u / N2;
        const int c = EPC == 1 ? u : u - el * N2;
        i = c % N;
        j = c / N;
        active = t < EPC * G * N2;
        if (!active) el = d = 0;
    }
    __device__ __forceinline__ int column() const { return i + N * j; }   // point index and place at k = 0
    // first place of the thread's line along direction dir (0 r, 1 s, 2 t)
    __device__ __forceinline__ int line(int dir) const {
        return dir == 0 ? N * j + fx_layer(N) * i : i + (dir == 1 ? fx_layer(N) : N) * j;
    }
    __device__ __forceinline__ int point(int kk) const { return G == 1 ? kk : d + G * kk; }
    __device__ __forceinline__ bool has(int kk) const { return G == 1 || N % G == 0 || d + G * kk < N; }
};

__device__ __forceinline__ FxConst fx_get(const FxConst *p) {
    const int4 q = *reinterpret_cast<const int4 *>(p);
    FxConst c;
    c.h = q.x;
    c.l = __int_as_float(q.y);
    c.f = __int_as_float(q.z);
    return c;
}
template <int M>
__device__ __forceinline__ fx::Acc fx_first(const FxTab<M> &t, int q, int xh, float xl, float xf) {
    const FxConst c = fx_get(t.v + q);
    return fx::first(c.h, c.l, c.f, xh, xl, xf);
}
template <int M>
__device__ __forceinline__ void fx_add(fx::Acc &a, const FxTab<M> &t, int q, int xh, float xl, float xf) {
    const FxConst c = fx_get(t.v + q);
    fx::add(a, c.h, c.l, c.f, xh, xl, xf);
}
__device__ __forceinline__ int2 fx_store(long long A, float B) {
    const fx::Pair p = fx::pair_of(A, B);
    return make_int2(p.h, __float_as_int(p.l));
}

// out(m) = sum_l M(m,l) v(l), plain or even-odd, handed to put(m, pair); the
// even-odd form gives m and N-1-m together.
template <int N, typename Put>
__device__ __forceinline__ void fx_line_plain(const int2 (&v)[N], const FxTab<N * N> &M, Put put) {
    float xf[N];
#pragma unroll
    for (int l = 0; l < N; l++) xf[l] = (float)v[l].x;
#pragma unroll
    for (int m = 0; m < N; m++) {
        fx::Acc acc = fx_first(M, m * N, v[0].x, __int_as_float(v[0].y), xf[0]);
        acc.A += fx::kHalf;
#pragma unroll
        for (int l = 1; l < N; l++) fx_add(acc, M, m * N + l, v[l].x, __int_as_float(v[l].y), xf[l]);
        put(m, fx_store(acc.A, acc.B));
    }
}

template <int N, typename Put>
__device__ __forceinline__ void fx_line_eo(const int2 (&v)[N], const FxEoHalf<N> &M, Put put) {
    constexpr int H = N / 2;
    int sh[H], dh[H];
    float sl[H], dl[H], sf[H], df[H];
#pragma unroll
    for (int l = 0; l < H; l++) {
        const float al = __int_as_float(v[l].y), bl = __int_as_float(v[N - 1 - l].y);
        sh[l] = v[l].x + v[N - 1 - l].x;
        dh[l] = v[l].x - v[N - 1 - l].x;
        sl[l] = al + bl;
        dl[l] = al - bl;
        sf[l] = (float)sh[l];
        df[l] = (float)dh[l];
    }
    const int ch = v[H].x;                       // the middle value (odd N)
    const float cl = __int_as_float(v[H].y), cf = (float)ch;
#pragma unroll
    for (int m = 0; m < H; m++) {
        fx::Acc P = fx_first(M.a, m * H, dh[0], dl[0], df[0]);
        P.A += fx::kHalf;
#pragma unroll
        for (int l = 1; l < H; l++) fx_add(P, M.a, m * H + l, dh[l], dl[l], df[l]);
        fx::Acc Q = fx_first(M.b, m * H, sh[0], sl[0], sf[0]);
#pragma unroll
        for (int l = 1; l < H; l++) fx_add(Q, M.b, m * H + l, sh[l], sl[l], sf[l]);
        if (N & 1) fx_add(Q, M.b, H * H + m, ch, cl, cf);
        put(m, fx_store(fx::wrap_add(P.A, Q.A), P.B + Q.B));
        put(N - 1 - m, fx_store(fx::wrap_sub(P.A, Q.A), P.B - Q.B));
    }
    if (N & 1) {
        fx::Acc Y = fx_first(M.c, 0, dh[0], dl[0], df[0]);
        Y.A += fx::kHalf;
#pragma unroll
        for (int l = 1; l < H; l++) fx_add(Y, M.c, l, dh[l], dl[l], df[l]);
        fx_add(Y, M.c, H, ch, cl, cf);
        put(H, fx_store(Y.A, Y.B));
    }
}

template <int N, bool EO, bool TR, int CP, typename Put>
__device__ __forceinline__ void fx_line(const int2 (&v)[N], const typename FxConsts<N, EO>::type &D, Put put) {
    if constexpr (EO)
        fx_line_eo<N>(v, TR ? D.bwd[CP] : D.fwd[CP], put);
    else
        fx_line_plain<N>(v, TR ? D.bwd[CP] : D.fwd[CP], put);
}

// A line from in to out; out may be in.
template <int N, bool EO, bool TR, int DIR>
__device__ __forceinline__ void fx_line_at(const int2 *in, int2 *out,
                                           const typename FxConsts<N, EO>::type &D) {
    constexpr int S = DIR == 0 ? 1 : (DIR == 1 ? N : fx_layer(N));
    int2 v[N];
#pragma unroll
    for (int l = 0; l < N; l++) v[l] = in[l * S];
    fx_line<N, EO, TR, DIR>(v, D, [&](int m, int2 y) { out[m * S] = y; });
}

// u = g w at one point: (ur, us, ut) from (wr, ws, wt) and the six factors
// (rr, rs), (rt, ss), (st, tt), shifted right by the point's s.
__device__ __forceinline__ void fx_contract(const int4 (&g4)[3], int2 &a, int2 &b, int2 &c) {
    const int2 g[6] = {make_int2(g4[0].x, g4[0].y), make_int2(g4[0].z, g4[0].w), make_int2(g4[1].x, g4[1].y),
                       make_int2(g4[1].z, g4[1].w), make_int2(g4[2].x, g4[2].y), make_int2(g4[2].z, g4[2].w)};
    // the factor 2^-32 of the small products' second half goes to the l of w
    const float al = __int_as_float(a.y) * 0x1p-32f, bl = __int_as_float(b.y) * 0x1p-32f,
                cl = __int_as_float(c.y) * 0x1p-32f;
    const float af = (float)a.x, bf = (float)b.x, cf = (float)c.x;
    const int s = g[0].y & 31;
    const float s2 = __int_as_float((127 - s) << 23);
    float gl[6], gf[6];
#pragma unroll
    for (int q = 0; q < 6; q++) {
        gl[q] = __int_as_float(g[q].y);
        gf[q] = (float)g[q].x;
    }
    auto row = [&](int q0, int q1, int q2) {
        fx::Acc u = fx::first(g[q0].x, gl[q0], gf[q0], a.x, al, af);
        fx::add(u, g[q1].x, gl[q1], gf[q1], b.x, bl, bf);
        fx::add(u, g[q2].x, gl[q2], gf[q2], c.x, cl, cf);
        return fx_store((u.A >> s) + fx::kHalf, u.B * s2);
    };
    const int2 u0 = row(0, 1, 2), u1 = row(1, 3, 4), u2 = row(2, 4, 5);
    a = u0;
    b = u1;
    c = u2;
}

// The operator's inner phases on the CTA's elements, by every thread: the
// forward derivatives of X along r and s into R and S and along t into TT
// (which may be X with G = 1); the contraction in place; the transposed
// derivatives in place.  With G = 1 the t lines and the contraction touch the
// thread's own column only.  Barriers between phases; none before the first
// and none after the last.  The pointers are the element's; g: its factors at
// the thread's column, [3][n^3].  on: the thread has a column of an element.
// s_low: with G = 3, the word that receives all ones if a t line is small (fx_note).
// Two points' factors are loaded ahead, the first before the barrier.  The
// loop over the points is not unrolled further: the straight-line code of an
// element did not fit the instruction cache.
template <int N, bool EO, int G>
__device__ __forceinline__ void fx_operator(const FxThread<N, G> &th, bool on, int2 *X, int2 *R, int2 *S, int2 *TT,
                                            const int4 *__restrict__ g, const typename FxConsts<N, EO>::type &D,
                                            unsigned *s_low) {
    constexpr int N2 = N * N, N3 = N * N * N, L = fx_layer(N), K = FxThread<N, G>::K;
    int4 gb[2][3];
    auto load = [&](int kk, int4 (&b)[3]) {
#pragma unroll
        for (int c = 0; c < 3; c++) b[c] = __ldcs(g + c * N3 + th.point(kk) * N2);
    };
    if (on) {
        if (G == 1 || th.d == 0) fx_line_at<N, EO, false, 0>(X + th.line(0), R + th.line(0), D);
        if (G == 1 || th.d == 1) fx_line_at<N, EO, false, 1>(X + th.line(1), S + th.line(1), D);
        if (G == 3 && th.d == 2) {
            int m = 0;                 // the magnitudes' bits
#pragma unroll
            for (int k = 0; k < N; k++) {
                const int h = X[th.line(2) + k * L].x;
                m |= h ^ (h >> 31);
            }
            fx_line_at<N, EO, false, 2>(X + th.line(2), TT + th.line(2), D);
            if (m != 0 && m < 1 << (30 - fx_grade(N))) *s_low = ~0u;
        }
        if (th.has(0)) load(0, gb[0]);     // n = 2 with G = 3: the third thread owns no point
        if (K > 1 && th.has(1)) load(1, gb[1]);
    }
    __syncthreads();
    if (on) {
        if (G == 1) fx_line_at<N, EO, false, 2>(X + th.line(2), TT + th.line(2), D);
        const int at = th.column();
        int2 *r = R + at, *s = S + at, *tt = TT + at;
        auto point = [&](int kk, int u) {
            if (!th.has(kk)) return;
            const int k = th.point(kk) * L;
            int2 a = r[k], b = s[k], c = tt[k];
            fx_contract(gb[u], a, b, c);
            r[k] = a;
            s[k] = b;
            tt[k] = c;
            if (kk + 2 < K && th.has(kk + 2)) load(kk + 2, gb[u]);
        };
#pragma unroll 1
        for (int kk = 0; kk + 1 < K; kk += 2) {
            point(kk, 0);
            point(kk + 1, 1);
        }
        if (K % 2) point(K - 1, 0);
        if (G == 1) fx_line_at<N, EO, true, 2>(TT + th.line(2), TT + th.line(2), D);
    }
    __syncthreads();
    if (on) {
        if (G == 1 || th.d == 0) fx_line_at<N, EO, true, 0>(R + th.line(0), R + th.line(0), D);
        if (G == 1 || th.d == 1) fx_line_at<N, EO, true, 1>(S + th.line(1), S + th.line(1), D);
        if (G == 3 && th.d == 2) fx_line_at<N, EO, true, 2>(TT + th.line(2), TT + th.line(2), D);
    }
}

// The sum of the three partials at a place.
__device__ __forceinline__ fx::Pair fx_sum(const int2 *R, const int2 *S, const int2 *TT, int at) {
    const int2 a = R[at], b = S[at], c = TT[at];
    fx::Pair p;
    p.h = a.x + b.x + c.x;
    p.l = __int_as_float(a.y) + __int_as_float(b.y) + __int_as_float(c.y);
    return p;
}

// The largest biased exponent of an element's input: every thread's maximum of
// the magnitudes' top words goes into the element's word of s_max (which is 0
// before); the caller synchronises, then reads it with fx_emax.
// The element's second word, s_max[EPC + el], says whether a column is small
// (fx_note).  G = 1: it holds the smallest of the columns' maxima, zeros left
// out, complemented; with one element per CTA it comes from the warps here, with
// several from the threads that find theirs small once the element's is known
// (fx_mark_small: a second atomic or warp reduction per element cost a CG iteration
// 2 to 4 % at n = 4, 6 and 9, a register across the barrier 1 to 2 % at n = 10).
// G = 3: the threads of the t lines mark it (fx_operator).
template <int N, int G>
__device__ __forceinline__ void fx_max_in(const FxThread<N, G> &th, bool on, unsigned top, unsigned *s_max) {
    constexpr int EPC = fx_epc(N, G);
    top = on ? top : 0u;
    if constexpr (EPC == 1) {
        const unsigned a = __reduce_max_sync(0xffffffffu, top);
        const unsigned l = G == 1 ? __reduce_max_sync(0xffffffffu, top ? ~top : 0u) : 0u;
        if ((threadIdx.x & 31) == 0) {
            atomicMax(s_max, a);
            if (G == 1) atomicMax(s_max + 1, l);
        }
    } else if constexpr (N >= 6) {      // a warp's threads belong to at most two elements
        const int first = (int)(threadIdx.x & ~31u) / (N * N);
        const unsigned a = __reduce_max_sync(0xffffffffu, th.el == first ? top : 0u);
        const unsigned b = __reduce_max_sync(0xffffffffu, th.el == first ? 0u : top);
        if ((threadIdx.x & 31) == 0) {
            if (first < EPC) atomicMax(s_max + first, a);
            if (first + 1 < EPC) atomicMax(s_max + first + 1, b);
        }
    } else {
        if (on) atomicMax(s_max + th.el, top);
    }
}

// x += xa p (the owed update, xa != 0), p = r + beta p and v = p on a thread's
// points; the pointers are the column's.  All loads of a step are issued before
// its stores: the compiler may not move a load over a store that might alias
// it, and one point at a time exposes the memory latency every time.
template <int N, bool JACOBI, int G>
__device__ __forceinline__ void fx_direction(const FxThread<N, G> &th, const double *r, double *p, double *x,
                                             const double *minv, double beta, double xa,
                                             double (&v)[FxThread<N, G>::K]) {
    constexpr int N2 = N * N, K = FxThread<N, G>::K, STEPS = (K + 4) / 5, C = (K + STEPS - 1) / STEPS;
#pragma unroll
    for (int k0 = 0; k0 < K; k0 += C) {
        double pv[C], rv[C], xv[C];
#pragma unroll
        for (int u = 0; u < C; u++)
            if (k0 + u < K && th.has(k0 + u)) {
                const int q = th.point(k0 + u) * N2;
                pv[u] = p[q];
                rv[u] = JACOBI ? r[q] * minv[q] : r[q];
                if (xa != 0.0) xv[u] = __ldcs(x + q);
            }
#pragma unroll
        for (int u = 0; u < C; u++)
            if (k0 + u < K && th.has(k0 + u)) {
                const int q = th.point(k0 + u) * N2;
                v[k0 + u] = fma(beta, pv[u], rv[u]);
                p[q] = v[k0 + u];
                if (xa != 0.0) __stcs(x + q, fma(xa, pv[u], xv[u]));
            }
    }
}

// The largest top word (sign off) of a thread's values.
template <int N, int G>
__device__ __forceinline__ unsigned fx_top_of(const FxThread<N, G> &th, const double (&v)[FxThread<N, G>::K]) {
    unsigned top = 0;
#pragma unroll
    for (int k = 0; k < FxThread<N, G>::K; k++) {
        const unsigned t = th.has(k) ? (unsigned)__double2hiint(v[k]) & 0x7fffffffu : 0u;
        top = t > top ? t : top;
    }
    return top;
}
__device__ __forceinline__ int fx_emax(unsigned top) {
    const int e = (int)(top >> 20);
    return e < fx::kMinExp ? fx::kMinExp : (e == 0x7ff ? fx::kNotFinite : e);
}
__device__ __forceinline__ int2 fx_input(double v, int emax) {
    const fx::Pair p = fx::from_double(v, emax);
    return make_int2(p.h, __float_as_int(p.l));
}

// The pairs of a thread's values into its column of X.
template <int N, int G>
__device__ __forceinline__ void fx_put_input(const FxThread<N, G> &th, const double (&v)[FxThread<N, G>::K], int emax,
                                             int2 *X) {
#pragma unroll
    for (int k = 0; k < FxThread<N, G>::K; k++)
        if (th.has(k)) X[th.column() + th.point(k) * fx_layer(N)] = fx_input(v[k], emax);
}

// Is point k of the thread's column on a face of the box?  cf: the faces of
// (i, j) that are on the box (fx_column_faces and box_faces), bf: box_faces.
template <int N, int G>
__device__ __forceinline__ unsigned fx_column_faces(const FxThread<N, G> &th) {
    return (unsigned)(th.i == 0) | ((unsigned)(th.i == N - 1) << 1) | ((unsigned)(th.j == 0) << 2) |
           ((unsigned)(th.j == N - 1) << 3);
}
template <int N>
__device__ __forceinline__ bool fx_on_face(unsigned cf, unsigned bf, int k) {
    return cf || (k == 0 && (bf & 16u)) || (k == N - 1 && (bf & 32u));
}

// The points k of the thread's column that are not on a face of the box, as bits.
template <int N, int G>
__device__ __forceinline__ unsigned fx_inner_points(const FxThread<N, G> &th, unsigned bf) {
    const unsigned all = (1u << N) - 1u;
    return (fx_column_faces(th) & bf) ? 0u : all & ~((bf >> 4) & 1u) & ~(((bf >> 5) & 1u) << (N - 1));
}

// The final pass of a CG head on a thread's points: w = the sum of the
// partials in FP64, box faces zeroed; the points' products w p of the
// fixed-point pairs, summed exactly over at most four points, go to
// flush(A, B) as (A + B) 2^(so + emax - 1052).  w, p: the column's.
template <int N, int G, typename Flush>
__device__ __forceinline__ void fx_final(const FxThread<N, G> &th, const int2 *X, const int2 *R, const int2 *S,
                                         const int2 *TT, double *w, const double *p, int so, int emax, unsigned bf,
                                         Flush flush) {
    constexpr int N2 = N * N, L = fx_layer(N), K = FxThread<N, G>::K;
    const int at = th.column();
    const unsigned cf = fx_column_faces(th) & bf;
    fx::Scale out;
    out.set(so);
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += 4) {
        long long dA = 0;
        float dB = 0.f;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            if (k0 + u >= K || !th.has(k0 + u)) break;
            const int k = th.point(k0 + u);
            fx::Pair s = fx_sum(R, S, TT, at + k * L);
            if (fx_on_face<N>(cf, bf, k)) {
                s.h = 0;
                s.l = 0.f;
            }
            const int2 x = fx_keep(N, G) ? X[at + k * L] : fx_input(p[k * N2], emax);
            dA += (long long)s.h * x.x;      // below 1.5 2^60 each: four of them fit
            dB = fmaf(s.l, (float)x.x, fmaf((float)s.h, __int_as_float(x.y), dB));
            w[k * N2] = out(s);
        }
        flush(dA, dB);
    }
    if (out.rest != 0) {
        const double post = out.post();
#pragma unroll 1
        for (int k = 0; k < K; k++)
            if (th.has(k)) w[th.point(k) * N2] *= post;
    }
}

// Graded elements.  A pair holds 54 bits below the element's largest entry, a
// floating-point value the same number below its own.  So a point all of whose
// inputs lie far below that entry loses as many bits here, and an element that
// has such a point is computed again in double-float arithmetic (fx_redo_list),
// which keeps 47 bits of every value.  The inputs of a point are above all those
// on the three lines through it (the operator's leading terms).  A line is small
// if its entries' exponents are all 8 or more below the element's largest (below
// 2^-8 to 2^-7 of it; more at n = 2 and 3, whose lines have too few entries to
// tell, fx_grade), and so is every line along a direction whose factors are below
// 2^-14 of the element's largest (sides 128 : 1; with t such a direction all
// elements are listed, and at 2^-6 flat boxes of 16 layers to one ran 11 to 18 %
// slower).  A point is small if all three lines through it are, leaving out
// lines of zeros along t (on a face of the box, where a field vanishes) and
// points on the box's faces, which the CG heads zero.  An element is graded if
// more than 1/64 of its points are small, or the lines through one are all below
// 2^-16: the few points beside the corners of a box where a smooth field vanishes
// (2^-8 at n = 8, 2^-14 at n = 16) are not worth another pass, whose latency is
// that of the whole call on small boxes (64 elements at n = 8 12.3 us
// instead of 8.2, of which 2 are the look at them).  And it is graded if all its entries are tiny (kMinExp), or its
// word says so.
// Why 8: on elements stretched by factors up to 100 and nine kinds of data
// (emulated, n = 2 to 16) the largest error of a kept element is mostly below the
// double-float operator's and at most 18 times as large (a single entry 2^7
// above the others); without the rule it is up to 250 times.  And among 50000
// elements of the directions of CG solves no column was small (n = 4 to 10).
// A CTA lists elements that may be graded on the way (fx_note) and looks at them
// again when it has done its share: with the test and the call inside the loop
// over the elements the loop itself ran 2 to 5 % slower.  A graded element costs
// three times another: 4096 of them at n = 10 take 262 us, others 80; in
// double-float arithmetic alone they all took 119.
// An element's word (ge): its exponent in the low 16 bits; kFxGraded: always
// computed again (fx_factors_kernel); then one bit per direction with small
// factors.
constexpr int kFxExp = 0xffff, kFxGraded = 1 << 16, kFxWeak = 1 << 17;
// The bits that put an element on the list whatever its input.
constexpr int kFxSpecial = kFxGraded | (kFxWeak << 2);
// The shift s of a point's factors (Scales) reaches about 2.4 log2(n) on a regular
// element; an element where it is 5 more is graded.
__host__ __device__ constexpr int fx_max_shift(int n) {
    return 5 + (n < 3 ? 2 : (n < 4 ? 3 : (n < 6 ? 4 : (n < 8 ? 6 : (n < 10 ? 7 : (n < 13 ? 8 : 9))))));
}

// The factors of the elements, whole arrays, and what graded elements need.
struct FxData {
    const int4 *g;      // pairs [E][3][n^3], two per entry
    const int *ge;      // the elements' words [E]
    const double *gd;   // gxyz [E][6][n^3]
    const void *dd;     // D in double-float pairs (DfConsts<N, EO>)
    int gexp;           // biased exponent of max|gxyz|
    int special;        // some element's word has one of kFxSpecial's bits
    int2 *list;         // scratch [E]: the CG heads' lists (FxList)
};

// A CTA's list of elements that may be graded.  CHAIN (the CG heads, whose CTAs
// take many groups): a chain through the scratch, an entry holding the element
// before (-1: none) and the exponent of the input; head: the last one listed.
// Otherwise (MODE 0: one group per CTA) the group's own slots, (element or -1,
// exponent), so that the operator alone keeps no state between or beside its launches;
// head >= 0: there is one.
template <int EPC, bool CHAIN>
struct FxList {
    int head;
    int2 slot[CHAIN ? 1 : EPC];
    __device__ __forceinline__ void init() {
        if (threadIdx.x == 0) head = -1;
        if (!CHAIN && threadIdx.x < EPC) slot[threadIdx.x].x = -1;
    }
};
// Puts an element on it, by one thread.
template <int EPC, bool CHAIN>
__device__ __noinline__ void fx_list(const FxData &fd, int64_t e, int64_t end, unsigned top,
                                     FxList<EPC, CHAIN> &list) {
    if (e >= end || top == 0u) return;
    if (CHAIN) {
        fd.list[e] = make_int2(atomicExch(&list.head, (int)e), (int)(top >> 20));
    } else {
        list.slot[CHAIN ? 0 : threadIdx.x] = make_int2((int)e, (int)(top >> 20));
        list.head = 0;
    }
}
// With several elements in a CTA, or G = 3: a thread whose column is small marks
// its element (fx_max_in).  With G = 3 it knows a third of the column only and
// marks what the t lines do not see, entries whose integer is 0.
template <int N, int G>
__device__ __forceinline__ void fx_mark_small(const FxThread<N, G> &th, const FxData &fd, bool on, unsigned top,
                                              unsigned elem, unsigned *s_max) {
    if (on && top && (top + (unsigned)((G == 1 ? fx_grade(N) : 30) << 20) <= elem || elem < kFxTiny || fd.special))
        s_max[fx_epc(N, G) + th.el] = ~0u;
}
// The list's upkeep, by the thread of each element of the CTA's group (e0, element
// threadIdx.x): top is the element's first word of s_max, s_low the second ones,
// which it clears.  The comparisons are all that an element costs that is not listed.
template <int N, int G, bool CHAIN>
__device__ __forceinline__ void fx_note(const FxData &fd, int64_t e0, int64_t end, unsigned top, unsigned *s_low,
                                        FxList<fx_epc(N, G), CHAIN> &list) {
    const unsigned low = s_low[threadIdx.x];
    bool may;
    if (fx_epc(N, G) > 1 || G == 3) {
        may = low != 0u;
        if (may) s_low[threadIdx.x] = 0;
    } else {
        s_low[threadIdx.x] = 0;
        may = low >= ~(top - (unsigned)(fx_grade(N) << 20)) || top < kFxTiny || fd.special;
    }
    if (may) fx_list(fd, e0 + threadIdx.x, end, top, list);
}

// One line of a graded element, one copy of its code: inlined, the lines would
// share the entries of D they load, in spilled registers.
template <int N, bool EO>
__device__ __noinline__ void fx_redo_line(const float2 *in, float2 *out, int base, int stride,
                                          const typename DfConsts<N, EO>::type *__restrict__ D, bool tr) {
    if constexpr (EO) line_eo<N>(in, out, base, stride, tr ? D->bwd : D->fwd);
    else line_plain<N>(in, out, base, stride, tr ? D->bwd : D->fwd);
}

// The points of a thread's column through which the lines along all three directions
// are small, of the `points` (bits): how many, or kFxFar if the lines through one are
// all 2^-16 of the largest entry or less.  X: the element's input in float pairs,
// its largest entry in [1, 2).  weak: bits of directions whose lines all are small.
constexpr int kFxFar = 1 << 12;     // more than 1/64 of an element; 64 times all threads' sum fits an int
template <int N, int G>
__device__ __forceinline__ int fx_small_points(const FxThread<N, G> &th, const float2 *X, int weak, unsigned points) {
    constexpr int L = fx_layer(N);
    constexpr float kSmall = 2.f / (1 << fx_grade(N));
    auto top = [&](int dir, int at, int stride) {
        float m = 0.f;
#pragma unroll
        for (int l = 0; l < N; l++) m = fmaxf(m, fabsf(X[at + l * stride].x));
        return (weak >> dir) & 1 ? 0.f : m;
    };
    const float t = top(2, th.column(), L);
    if (t >= kSmall || (t == 0.f && !((weak >> 2) & 1))) return 0;      // a line of zeros does not count
    int count = 0;
#pragma unroll 1
    for (int k = 0; k < N; k++) {
        if (!((points >> k) & 1u)) continue;
        const float m = fmaxf(t, fmaxf(top(0, N * th.j + L * k, 1), top(1, th.i + L * k, N)));
        if (m < 0x1p-15f) return kFxFar;
        count += m < kSmall;
    }
    return count;
}

// A CTA's list, when it has done its share: w = ax_e(v) in double-float arithmetic
// on those listed elements that are graded, zero on the box's faces if `mask`.
// The layout and the phases are fx_operator's, the line products and scales
// (an element's largest exponent, max|gxyz|) the double-float head's.  The sums
// <w,p>_c keep the fixed-point products, whose error the large entries set.
// Every thread calls it; sm holds the CTA's arrays, arrays of them per element.
template <int N, bool EO, int G, bool CHAIN>
__device__ __noinline__ void fx_redo_list(const FxData &fd, const FxList<fx_epc(N, G), CHAIN> &list, const double *v,
                                          double *w, bool mask, const Mesh &m, int2 *sm, int arrays) {
    constexpr int N2 = N * N, N3 = N * N * N, A = fx_array(N), L = fx_layer(N), K = FxThread<N, G>::K;
    constexpr int EPC = fx_epc(N, G);
    __shared__ int2 s_slot[EPC];       // the elements at work and their exponents
    __shared__ int s_next;
    __shared__ int s_small[EPC];       // their small points (fx_small_points)
    FxThread<N, G> th;
    th.init();
    const auto *D = (const typename DfConsts<N, EO>::type *)fd.dd;
    float2 *X = (float2 *)sm + arrays * A * th.el, *R = X + A, *S = X + 2 * A, *TT = arrays == 4 ? X + 3 * A : X;
    const int at = th.column();
    auto line = [&](const float2 *in, float2 *out, int dir, bool tr) {
        fx_redo_line<N, EO>(in, out, th.line(dir), dir == 0 ? 1 : (dir == 1 ? N : L), D, tr);
    };
    int head = list.head;
    // a chain has an element at most once; the bound ends the walk whatever it holds
    for (int64_t left = m.E; head >= 0 && left > 0; head = s_next, left--) {
        __syncthreads();               // the arrays and the shared words are free
        if (threadIdx.x == 0) {
            int e = head;
            for (int el = 0; el < EPC; el++) {
                if (!CHAIN) {
                    s_slot[el] = list.slot[CHAIN ? 0 : el];
                    continue;
                }
                s_slot[el] = make_int2(e, 0);
                if (e < 0) continue;
                const int2 entry = fd.list[e];
                s_slot[el].y = entry.y;
                e = entry.x;
            }
            s_next = CHAIN ? e : -1;
        }
        if (threadIdx.x < EPC) s_small[threadIdx.x] = 0;
        __syncthreads();
        const int64_t e = s_slot[th.el].x;
        const int emax = s_slot[th.el].y;
        const int word = e >= 0 ? fd.ge[e] : 0;
        const int64_t q0 = e * N3 + at;
        // not finite: the results are NaN already
        bool on = th.active && e >= 0 && emax != 0x7ff && !(word & fx::kNotFinite);
        unsigned bf = 0;
        if (mask && on) {
            int ex, ey, ez;
            element_coords(e, m, ex, ey, ez);
            bf = box_faces(ex, ey, ez, m);
        }
        if (on) {
            double x[K];
#pragma unroll
            for (int kk = 0; kk < K; kk++)
                if (th.has(kk)) x[kk] = v[q0 + th.point(kk) * N2];
#pragma unroll
            for (int kk = 0; kk < K; kk++)
                if (th.has(kk)) X[at + th.point(kk) * L] = dfa::split_scaled(x[kk], 1023 - emax);
        }
        __syncthreads();
        if (on) {
            const int small = (word & kFxGraded) || emax <= fx::kMinExp
                                  ? kFxFar
                                  : fx_small_points(th, X, word / kFxWeak, fx_inner_points(th, bf));
            if (small) atomicAdd(&s_small[th.el], small);
        }
        __syncthreads();
        // G = 3: a column's threads count its points three times
        on = on && s_small[th.el] * 64 > G * N3;
        if (on) {
            if (G == 1 || th.d == 0) line(X, R, 0, false);
            if (G == 1 || th.d == 1) line(X, S, 1, false);
            if (G == 3 && th.d == 2) line(X, TT, 2, false);
        }
        __syncthreads();
        if (on) {
            if (G == 1) line(X, TT, 2, false);
            const double *g = fd.gd + e * 6 * N3 + at;
            double gv[2][6];            // a point's factors are loaded while the one before is contracted
            auto load = [&](int kk) {
#pragma unroll
                for (int c = 0; c < 6; c++) gv[kk & 1][c] = g[(int64_t)c * N3 + th.point(kk) * N2];
            };
            if (th.has(0)) load(0);
#pragma unroll 2
            for (int kk = 0; kk < K; kk++) {
                if (!th.has(kk)) break;
                if (kk + 1 < K && th.has(kk + 1)) load(kk + 1);
                const int q = at + th.point(kk) * L;
                float2 f[6];
#pragma unroll
                for (int c = 0; c < 6; c++) f[c] = dfa::split_near(gv[kk & 1][c], 1023 - fd.gexp);
                df_contract(f, R[q], S[q], TT[q]);
            }
            if (G == 1) line(TT, TT, 2, true);
        }
        __syncthreads();
        if (on) {
            if (G == 1 || th.d == 0) line(R, R, 0, true);
            if (G == 1 || th.d == 1) line(S, S, 1, true);
            if (G == 3 && th.d == 2) line(TT, TT, 2, true);
        }
        __syncthreads();
        if (on) {
            const unsigned cf = fx_column_faces(th) & bf;
#pragma unroll 1
            for (int kk = 0; kk < K; kk++) {
                if (!th.has(kk)) break;
                const int k = th.point(kk), q = at + k * L;
                const double wv = dfa::join_scaled(dfa::add(dfa::add(R[q], S[q]), TT[q]),
                                                   (emax - 1023) + (fd.gexp - 1023));
                w[q0 + k * N2] = fx_on_face<N>(cf, bf, k) ? 0.0 : wv;
            }
        }
    }
}

// Arguments of fx_elements (whole arrays).
struct FxIO {
    const double *u;    // MODE 0: input
    const double *r;    // MODE 1: residual
    double *p;          // MODE 1: search direction (updated in place)
    double *x;          // MODE 1: iterate (owed update applied when xa != 0)
    const double *minv; // MODE 1: Jacobi inverse diagonal (z = minv r), or null
    double *w;          // output
};

// ax_e on the elements e0 .. e0 + fx_epc(N, G) - 1 below e1, by the whole CTA
// (every thread must call it; it contains barriers).  sm holds the arrays
// without `keep`, s_max two words per element, 0 on entry and exit.  MODE 1 is
// the CG head of the forms that have their own kernels for the rest (Jacobi,
// mask array): x += xa p, p = z + beta p, w = ax_e(p); with fuse, box-face
// points of w are zeroed and the local products w p (p is continuous, so
// their sum over all points is the assembled product) are added to dot.
template <int N, int MODE, bool EO, int G>
__device__ __forceinline__ void fx_elements(const FxIO &io, const FxData &fd, int64_t e0, int64_t e1, double beta,
                                            double xa, bool fuse, const Mesh &m, const FxThread<N, G> &th,
                                            const typename FxConsts<N, EO>::type &D, int2 *sm, unsigned *s_max,
                                            FxList<fx_epc(N, G), MODE != 0> &list, double &dot) {
    constexpr int N2 = N * N, N3 = N * N * N, A = fx_array(N), L = fx_layer(N), K = FxThread<N, G>::K;
    constexpr int EPC = fx_epc(N, G);
    const int64_t e = e0 + th.el;
    const bool on = th.active && e < e1;
    int2 *X = sm + 3 * A * th.el, *R = X + A, *S = X + 2 * A, *TT = G == 3 ? X + 3 * A : X;
    const int64_t q0 = e * N3 + th.column();
    const int at = th.column();
    double v[K];
    unsigned top = 0;
    if (on) {
        if (MODE == 0) {
#pragma unroll
            for (int k = 0; k < K; k++)
                if (th.has(k)) v[k] = __ldg(io.u + q0 + th.point(k) * N2);
        } else if (io.minv) {
            fx_direction<N, true>(th, io.r + q0, io.p + q0, io.x + q0, io.minv + q0, beta, xa, v);
        } else {
            fx_direction<N, false>(th, io.r + q0, io.p + q0, io.x + q0, nullptr, beta, xa, v);
        }
        top = fx_top_of(th, v);
    }
    fx_max_in(th, on, top, s_max);
    __syncthreads();
    const unsigned elem = s_max[th.el];
    const int emax = fx_emax(elem);
    if (EPC > 1 || G == 3) fx_mark_small(th, fd, on, top, elem, s_max);
    if (on) fx_put_input(th, v, emax, X);
    __syncthreads();
    unsigned etop = 0;
    if (threadIdx.x < EPC) {
        etop = s_max[threadIdx.x];
        s_max[threadIdx.x] = 0;
    }
    // loaded here: after the operator its latency showed (504 elements at n = 16
    // 52.4 us instead of 51.3)
    const int ge = on ? fd.ge[e] & kFxExp : 0;
    fx_operator<N, EO>(th, on, X, R, S, TT, fd.g + e * 3 * N3 + th.column(), D, s_max + EPC);
    if (threadIdx.x < EPC) fx_note<N, G>(fd, e0, e1, etop, s_max + EPC, list);
    __syncthreads();
    if (on) {
        fx::Scale out;
        out.set(emax + ge + D.so0);
        unsigned bf = 0;
        if (MODE == 1 && fuse) {
            int ex, ey, ez;
            element_coords(e, m, ex, ey, ez);
            bf = box_faces(ex, ey, ez, m);
        }
        const unsigned cf = fx_column_faces(th) & bf;
#pragma unroll 4
        for (int kk = 0; kk < K; kk++) {
            if (!th.has(kk)) break;
            const int k = th.point(kk);
            const double wv = out(fx_sum(R, S, TT, at + k * L));
            io.w[q0 + k * N2] = MODE == 1 && fuse && fx_on_face<N>(cf, bf, k) ? 0.0 : wv;
        }
        if (out.rest != 0) {
            const double post = out.post();
#pragma unroll 1
            for (int kk = 0; kk < K; kk++)
                if (th.has(kk)) io.w[q0 + th.point(kk) * N2] *= post;
        }
        if (MODE == 1 && fuse) {
#pragma unroll 4
            for (int kk = 0; kk < K; kk++) {
                if (!th.has(kk)) break;
                dot = fma(io.w[q0 + th.point(kk) * N2], io.p[q0 + th.point(kk) * N2], dot);
            }
        }
    }
    // no barrier: a thread's next input goes to X, which no other thread reads
    // any more after the forward products (with G = 1 but itself), and the two
    // barriers before the next forward products protect R, S and TT
}

// ------------------------------------------------------------------ set-up
// The scales of D (row major, FP64): c and rho per row index, kf, kb and the
// power of two that remains.
struct FxScales {
    double c[kMaxN], rho[kMaxN], kf, kb;
    int so0;
};
struct FxRows {
    double rho[kMaxN];
};

// The largest k with max |row sum| k <= 2^32 and max |entry| k < 2^31.
inline double fx_matrix_scale(const double *D, const double *c, int n, bool tr) {
    double rs = 0.0, mx = 0.0;
    for (int i = 0; i < n; i++) {
        double s = 0.0;
        for (int l = 0; l < n; l++) {
            const double v = fabs(tr ? D[l * n + i] * c[l] : D[i * n + l] * c[i]);
            s += v;
            mx = fmax(mx, v);
        }
        rs = fmax(rs, s);
    }
    return mx > 0.0 ? fmin(4294967296.0 / rs, 2147483648.0 / mx) * (1.0 - 1e-8) : 1.0;
}

inline FxScales fx_scales(const double *D, int n) {
    FxScales S{};
    double R[kMaxN], lo = 0.0;
    for (int i = 0; i < n; i++) {
        R[i] = 0.0;
        for (int l = 0; l < n; l++) R[i] += fabs(D[i * n + l]);
    }
    for (int i = 0; i < n; i++) {
        const double v = fmax(R[i], R[n - 1 - i]);   // the same for both rows of an even-odd pair
        if (v > 0.0 && (lo == 0.0 || v < lo)) lo = v;
    }
    for (int i = 0; i < n; i++) {
        const double v = fmax(R[i], R[n - 1 - i]);
        S.c[i] = v > 0.0 ? pow(v / lo, -0.75) : 1.0;
    }
    S.kf = fx_matrix_scale(D, S.c, n, false);
    S.kb = fx_matrix_scale(D, S.c, n, true);
    int ef, eb;
    const double mu = frexp(S.kf, &ef) * frexp(S.kb, &eb);
    S.so0 = -(ef + eb) - 2009;
    for (int i = 0; i < n; i++) S.rho[i] = 1.0 / (S.c[i] * sqrt(mu));
    return S;
}

inline FxRows fx_rows(const FxScales &S) {
    FxRows r;
    for (int i = 0; i < kMaxN; i++) r.rho[i] = S.rho[i];
    return r;
}

// The scale of a point's six scaled factors v (rr, rs, rt, ss, st, tt): the
// exponent eq with which the largest absolute row sum of the 3 x 3 matrix
// lies in (2^30, 2^31], in units of 2^(eq - 1053).  ex: the factors' biased
// exponents (0: the factor counts as 0).  kNotFinite if one of them is NaN or Inf.
__device__ __forceinline__ int fx_point_exponent(const double (&v)[6], int (&ex)[6]) {
    int e0 = 0;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        ex[c] = (int)((__double_as_longlong(v[c]) >> 52) & 0x7ff);
        e0 = ex[c] > e0 ? ex[c] : e0;
    }
    if (e0 == 0x7ff) return fx::kNotFinite;
    unsigned long long m[6];   // magnitudes rounded up, 31 bits for the largest
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v[c]);
        const int sh = 22 + e0 - ex[c];
        m[c] = ex[c] == 0 ? 0ull
                          : (((b & 0xfffffffffffffull) | 0x10000000000000ull) >> (sh < 63 ? sh : 63)) + 1ull;
    }
    const unsigned long long r0 = m[0] + m[1] + m[2], r1 = m[1] + m[3] + m[4], r2 = m[2] + m[4] + m[5];
    const unsigned long long r = r0 > r1 ? (r0 > r2 ? r0 : r2) : (r1 > r2 ? r1 : r2);
    return e0 + (r > 0x7ffffffcull) + (r > 0xfffffff8ull);
}

// The directions of an element whose factors are small everywhere: gd holds the
// largest biased exponents of its rr, ss and tt factors (the largest factor of a
// positive definite matrix is one of them).
__device__ __forceinline__ int fx_weak_bits(const int (&gd)[3]) {
    const int top = gd[0] > gd[1] ? (gd[0] > gd[2] ? gd[0] : gd[2]) : (gd[1] > gd[2] ? gd[1] : gd[2]);
    int bits = 0;
    for (int d = 0; d < 3; d++) bits |= gd[d] < top - 14 ? kFxWeak << d : 0;
    return bits;
}

// A point's factors with the row scales of D.
__device__ __forceinline__ void fx_scale_point(double (&v)[6], int q, int n, const FxRows &rows) {
    const double a = rows.rho[q % n], b = rows.rho[(q / n) % n], c = rows.rho[q / (n * n)];
    v[0] *= a * a;
    v[1] *= a * b;
    v[2] *= a * c;
    v[3] *= b * b;
    v[4] *= b * c;
    v[5] *= c * c;
}

// The pairs of a point's six scaled factors with exponents ex (fx_point_exponent)
// at an element exponent ge: (rr, rs), (rt, ss), (st, tt), the point's shift in
// the low bits of rr's float.
__device__ __forceinline__ void fx_point_pairs(const double (&v)[6], const int (&ex)[6], int eq, int ge, int4 (&o)[3]) {
    int s = ge - eq;
    s = s < 31 ? s : 31;
    int2 p[6];
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v[c]);
        int sh = ge - s - ex[c];
        sh = sh < 63 ? sh : 63;
        unsigned long long f = ex[c] == 0 ? 0ull : (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10) >> sh;
        f += 0x80000000ull;
        int h = (int)(f >> 32);
        float l = (float)(int)((unsigned)f ^ 0x80000000u) * 0x1p-64f;
        if (b >> 63) {
            h = -h;
            l = -l;
        }
        p[c] = make_int2(h, __float_as_int(l));
    }
    p[0].y = (p[0].y & ~31) | s;
#pragma unroll
    for (int c = 0; c < 3; c++) o[c] = make_int4(p[2 * c].x, p[2 * c].y, p[2 * c + 1].x, p[2 * c + 1].y);
}

// Does D lose precision in one scale?  Its pairs hold 55 bits below the largest
// absolute row sum; a row or a column all of whose entries lie more than 2^7
// below the largest entry keeps fewer than double-float pairs do.
inline bool fx_graded_matrix(const double *D, int n) {
    const FxScales S = fx_scales(D, n);
    double top = 0.0, row[kMaxN] = {}, col[kMaxN] = {};
    for (int i = 0; i < n; i++)
        for (int l = 0; l < n; l++) {
            const double v = fabs(D[i * n + l] * S.c[i]);
            row[i] = fmax(row[i], v);
            col[l] = fmax(col[l], v);
            top = fmax(top, v);
        }
    for (int i = 0; i < n; i++)
        if ((row[i] > 0.0 && row[i] < 0x1p-7 * top) || (col[i] > 0.0 && col[i] < 0x1p-7 * top)) return true;
    return false;
}

// Floats of D's double-float tables in either form (DfConsts).
constexpr int fx_df_floats(int n) { return 4 * n * n + 8 * (n + 1); }

// v k to entry q: the product's rounding error goes to l.
template <int M>
inline void fx_put(FxTab<M> &t, int q, double v, double k) {
    const double s = v * k, e = fma(v, k, -s), h = rint(s);
    t.v[q].h = (int)h;
    t.v[q].l = (float)ldexp((s - h) + e, -32);
    t.v[q].f = (float)ldexp(h, -32);
    t.v[q].pad = 0;
}

template <int N>
inline void fx_eo_half(const double *M, bool tr, double k, FxEoHalf<N> &E) {
    constexpr int H = N / 2;
    auto at = [&](int m, int l) { return tr ? M[l * N + m] : M[m * N + l]; };
    for (int m = 0; m < H; m++) {
        for (int l = 0; l < H; l++) {
            fx_put(E.a, m * H + l, 0.5 * (at(m, l) + at(N - 1 - m, l)), k);
            fx_put(E.b, m * H + l, 0.5 * (at(m, l) - at(N - 1 - m, l)), k);
        }
        fx_put(E.b, H * H + m, (N & 1) ? at(m, H) : 0.0, k);
    }
    for (int l = 0; l <= H; l++) fx_put(E.c, l, (N & 1) ? at(H, l) : 0.0, k);
}

template <int N, bool EO>
inline void fx_consts(const double *D, typename FxConsts<N, EO>::type &C) {
    const FxScales S = fx_scales(D, N);
    double M[N * N];
    for (int i = 0; i < N; i++)
        for (int l = 0; l < N; l++) M[i * N + l] = D[i * N + l] * S.c[i];
    C.so0 = S.so0;
    if constexpr (EO) {
        fx_eo_half<N>(M, false, S.kf, C.fwd[0]);
        fx_eo_half<N>(M, true, S.kb, C.bwd[0]);
    } else {
        for (int i = 0; i < N; i++)
            for (int l = 0; l < N; l++) {
                fx_put(C.fwd[0], i * N + l, M[i * N + l], S.kf);
                fx_put(C.bwd[0], i * N + l, M[l * N + i], S.kb);
            }
    }
    for (int d = 1; d < 3; d++) {
        C.fwd[d] = C.fwd[0];
        C.bwd[d] = C.bwd[0];
    }
}

}  // namespace nekgb
