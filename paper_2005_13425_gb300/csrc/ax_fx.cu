// Set-up and dispatch of the fixed-point ax_e (ax_fx_kernel.cuh; its kernels
// are instantiated in ax_fx_n*.cu, several sources so that they compile in
// parallel).
#include <math.h>

#include "ax_fx_core.cuh"

namespace nekgb {

template <int N>
nb_status launch_fx_n(nb_ctx *c, const double *u, double *w, int mode);
template <int N>
void fx_tables_n(nb_ctx *c);

// ---------------------------------------------------------------- set-up
// gxyz in fixed-point pairs (ax_fx_core.cuh, Scales), one CTA per element:
// first each point's exponent and their maximum ge, then the pairs.  The
// element's word (ax_fx_core.cuh, Graded elements): kFxGraded if a point's
// factors lie further below the element's largest than they do on a regular
// element of this order by 2^5 (measured with Jacobians graded up to 2^18: no
// larger error than the double-float operator's relative to max|w|, and up to
// 2^7 times as large relative to the point's own terms), or all_graded.
__global__ void __launch_bounds__(256)
fx_factors_kernel(const double *__restrict__ x, int4 *__restrict__ y, int *__restrict__ ge, int64_t E, int n,
                  FxRows rows, bool all_graded, int *special) {
    const int n3 = n * n * n;
    __shared__ int s_ge, s_low, s_gd[3];
    for (int64_t e = blockIdx.x; e < E; e += gridDim.x) {
        const double *g = x + e * 6 * n3;
        auto point = [&](int q, double (&v)[6], int (&ex)[6]) {
#pragma unroll
            for (int c = 0; c < 6; c++) v[c] = g[(int64_t)c * n3 + q];
            fx_scale_point(v, q, n, rows);
            return fx_point_exponent(v, ex);
        };
        double v[6];
        int ex[6], top = 0, low = 1 << 20, gd[3] = {0, 0, 0};
        __syncthreads();
        if (threadIdx.x == 0) {
            s_ge = 0;
            s_low = 1 << 20;
            for (int d = 0; d < 3; d++) s_gd[d] = 0;
        }
        __syncthreads();
        for (int q = threadIdx.x; q < n3; q += blockDim.x) {
            const int eq = point(q, v, ex);
            top = eq > top ? eq : top;
            if (eq > 0) low = eq < low ? eq : low;      // 0: no factors at all
            for (int d = 0; d < 3; d++) {
                const int x = ex[d == 0 ? 0 : 2 * d + 1];
                gd[d] = x > gd[d] ? x : gd[d];
            }
        }
        atomicMax(&s_ge, top);
        atomicMin(&s_low, low);
        for (int d = 0; d < 3; d++) atomicMax(&s_gd[d], gd[d]);
        __syncthreads();
        top = s_ge;
        for (int q = threadIdx.x; q < n3; q += blockDim.x) {
            const int eq = point(q, v, ex);
            int4 o[3];
            fx_point_pairs(v, ex, eq, top, o);
#pragma unroll
            for (int c = 0; c < 3; c++) y[(e * 3 + c) * n3 + q] = o[c];
        }
        if (threadIdx.x == 0) {
            for (int d = 0; d < 3; d++) gd[d] = s_gd[d];
            const int word = top | fx_weak_bits(gd) | (all_graded || top - s_low > fx_max_shift(n) ? kFxGraded : 0);
            ge[e] = word;
            if (word & kFxSpecial) *special = 1;
        }
    }
}

// Largest binary exponent (biased) of |x| over an array.
__global__ void max_exponent_kernel(const double *__restrict__ x, int64_t n, int *out) {
    int emax = 0;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int ex = (int)((__double_as_longlong(x[q]) >> 52) & 0x7ff);
        emax = ex > emax ? ex : emax;
    }
    emax = __reduce_max_sync(0xffffffffu, emax);
    if ((threadIdx.x & 31) == 0) atomicMax(out, emax);
}

// The fixed-point scale of the CG head's exact <w,p>_c: S = dot_shift0 -
// e(<p,p>_c), e the binary exponent.  Every |w_q| is at most
// A max|p| with A = 9 |D|_1 |D|_inf max|G| (three derivatives, the 3x3
// contraction, three transposed derivatives), and max|p| <= sqrt(8 <p,p>_c),
// so a thread's share (at most four of its points) is below 32 A <p,p>_c.
// sa below takes 288 A (a further factor 9 of margin) and another 16x for
// the recursion's <p,p>_c, so the share stays below 2^(sa + e).  Summing the
// shares, at most 6 n^2 per element, then stays below 2^125 (dot_lim): no
// 128-bit sum overflows.  The grid of the sum, 2^-S, is 2^-dot_lim of that bound.
static int fx_dot_lim(const nb_ctx *c) {
    const int n = c->m.n;
    return 125 - (int)ceil(log2(8.0 * (double)c->m.E * n * n));
}

static int fx_dot_shift0(const nb_ctx *c) {
    const int n = c->m.n;
    double d1 = 0.0, dinf = 0.0;
    for (int i = 0; i < n; i++) {
        double rs = 0.0, cs = 0.0;
        for (int l = 0; l < n; l++) {
            rs += fabs(c->D_host[i * n + l]);
            cs += fabs(c->D_host[l * n + i]);
        }
        dinf = fmax(dinf, rs);
        d1 = fmax(d1, cs);
    }
    // max|G| < 2^(gexp - 1022)
    const int sa = (int)ceil(log2(288.0 * 9.0 * d1 * dinf)) + (c->gxyz_exp - 1022) + 1 + 4;
    return fx_dot_lim(c) - sa;
}

static void fx_tables(nb_ctx *c) {
    switch (c->m.n) {
#define NB_CASE(NN) case NN: fx_tables_n<NN>(c); break;
        NB_CASE(2) NB_CASE(3) NB_CASE(4) NB_CASE(5) NB_CASE(6) NB_CASE(7) NB_CASE(8)
        NB_CASE(9) NB_CASE(10) NB_CASE(11) NB_CASE(12) NB_CASE(13) NB_CASE(14) NB_CASE(15)
        NB_CASE(16)
#undef NB_CASE
    }
}

nb_status prepare_fx(nb_ctx *c) {
    c->d_eo = centro_antisymmetric(c->D_host, c->m.n);
    const int64_t ng = (int64_t)6 * c->m.n * c->m.n * c->m.n * c->m.E;
    const bool df = c->d_eo && df_head_elements(c->m.E, c->m.n);
    // one allocation: the pairs, the float pairs (few elements), the elements'
    // words, the largest exponent of the whole box and whether an element is
    // special, D in double-float pairs, the scratch of graded elements
    const size_t bytes = sizeof(int2) * (ng * (df ? 2 : 1) + c->m.E) + sizeof(int) * (c->m.E + 2) +
                         sizeof(float) * fx_df_floats(c->m.n);
    cudaError_t e = dev_alloc((void **)&c->d_gxyz_fx, bytes);
    if (e != cudaSuccess) return cuda_fail(e, "alloc gxyz pairs");
    c->device_bytes += bytes;
    if (df) c->d_gxyz_df = (float2 *)((int2 *)c->d_gxyz_fx + ng);
    c->d_redo_list = (int2 *)c->d_gxyz_fx + ng * (df ? 2 : 1);
    c->d_ge = (int *)(c->d_redo_list + c->m.E);
    int *d_ex = c->d_ge + c->m.E;
    c->d_D_df = (float *)(d_ex + 2);
    int found[2] = {0, 0};
    bool d_finite = true;
    for (int q = 0; q < c->m.n * c->m.n; q++) d_finite = d_finite && isfinite(c->D_host[q]);
    FxRows rows = fx_rows(fx_scales(c->D_host, c->m.n));
    // a D that is not finite has no fixed-point form: every element's factors
    // become "not finite" (and so its results), and the tables stay 0
    for (int i = 0; i < kMaxN && !d_finite; i++) rows.rho[i] = NAN;
    e = cudaMemsetAsync(d_ex, 0, sizeof found, c->stream);
    if (e == cudaSuccess) {
        const int64_t cap = (int64_t)device_sms() * 8;
        max_exponent_kernel<<<1024, 256, 0, c->stream>>>(c->d_gxyz, ng, d_ex);
        fx_factors_kernel<<<(int)(c->m.E < cap ? c->m.E : cap), 256, 0, c->stream>>>(c->d_gxyz, c->d_gxyz_fx, c->d_ge,
                                                                                c->m.E, c->m.n, rows,
                                                                                d_finite && fx_graded_matrix(c->D_host, c->m.n),
                                                                                d_ex + 1);
        e = cudaGetLastError();
    }
    fx_tables(c);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(c->d_D_df, c->df_tab.data(), sizeof(float) * c->df_tab.size(), cudaMemcpyHostToDevice,
                            c->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(found, d_ex, sizeof found, cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return cuda_fail(e, "gxyz pairs");
    int gexp = found[0];
    c->fx_special = found[1];
    c->op_finite = d_finite && gexp < 2047;
    gexp = gexp < 1 ? 1 : (gexp > 2046 ? 2046 : gexp);
    c->gxyz_exp = gexp;
    c->fx_dot_lim = fx_dot_lim(c);
    c->fx_dot_shift0 = c->op_finite ? fx_dot_shift0(c) : 0;
    return df ? prepare_df(c) : NB_OK;
}

// True when D(i,l) = -D(n-1-i, n-1-l) to rounding (GLL derivative matrices).
bool centro_antisymmetric(const double *D, int n) {
    double mx = 0.0, asym = 0.0;
    for (int q = 0; q < n * n; q++) mx = fmax(mx, fabs(D[q]));
    for (int i = 0; i < n; i++)
        for (int l = 0; l < n; l++)
            asym = fmax(asym, fabs(D[i * n + l] + D[(n - 1 - i) * n + (n - 1 - l)]));
    return asym <= 1e-14 * mx;
}

nb_status launch_ax_fx(nb_ctx *c, const double *u, double *w, int mode) {
    switch (c->m.n) {
#define NB_CASE(NN) case NN: return launch_fx_n<NN>(c, u, w, mode);
        NB_CASE(2) NB_CASE(3) NB_CASE(4) NB_CASE(5) NB_CASE(6) NB_CASE(7) NB_CASE(8)
        NB_CASE(9) NB_CASE(10) NB_CASE(11) NB_CASE(12) NB_CASE(13) NB_CASE(14) NB_CASE(15)
        NB_CASE(16)
#undef NB_CASE
    }
    return fail(NB_ERR_ARG, "unsupported n");
}

}  // namespace nekgb
