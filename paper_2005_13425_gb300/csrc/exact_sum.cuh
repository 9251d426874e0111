// Exact 128-bit fixed-point sums: <w,p>_c of the FP64 CG heads, whose dynamic
// element schedule must not change it.
#pragma once

#include "internal.cuh"
#include "reduce.cuh"

namespace nekgb {

using u128 = unsigned __int128;

__device__ __forceinline__ u128 shfl_down_u128(u128 v, int o) {
    const unsigned long long lo = __shfl_down_sync(0xffffffffu, (unsigned long long)v, o);
    const unsigned long long hi = __shfl_down_sync(0xffffffffu, (unsigned long long)(v >> 64), o);
    return ((u128)hi << 64) | lo;
}

// Sum over the CTA (modulo 2^128, i.e. exact for the signed values the head
// produces); the total is valid in thread 0.  red: 2 * (warps) doubles.
__device__ __forceinline__ u128 block_sum_u128(u128 v, double *red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += shfl_down_u128(v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) {
        red[2 * wid] = __longlong_as_double((long long)(unsigned long long)(v >> 64));
        red[2 * wid + 1] = __longlong_as_double((long long)(unsigned long long)v);
    }
    __syncthreads();
    u128 t = 0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); k++)
            t += ((u128)(unsigned long long)__double_as_longlong(red[2 * k]) << 64) |
                 (unsigned long long)__double_as_longlong(red[2 * k + 1]);
    return t;
}

// x 2^k for any k (two exact power-of-two factors).
__device__ __forceinline__ double scale_pow2(double x, int k) {
    const int k1 = k / 2, k2 = k - k1;
    return x * __longlong_as_double((long long)(k1 + 1023) << 52) * __longlong_as_double((long long)(k2 + 1023) << 52);
}

// Is <p,p>_c finite?  The integer sum cannot carry a NaN or an Inf of p, so a head
// ends the solve when this does not hold (or the operator's data is not finite).
__device__ __forceinline__ bool finite_pp(double pn) {
    return (int)((__double_as_longlong(pn) >> 52) & 0x7ff) != 0x7ff;
}

// The sums of a head's threads (at the scale 2^S) over the CTA, and by the last
// CTA over all of them; that CTA forms alpha.  Every thread must call it.  red:
// 32 doubles of shared memory (as many as 2 per warp).
__device__ __forceinline__ void finish_exact_sum(CgScalars *sc, double *partials, u128 mine, int S, bool out_of_range,
                                                 bool finite, double *red) {
    const int range_fault = __syncthreads_or(out_of_range);
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        if (range_fault || !finite) {   // seen by the last CTA's finalize_alpha, which ends the solve
            if (finite) sc->fault = kFaultExactSumRange;
            sc->status = (int)NB_ERR_BREAKDOWN;
        }
        partials[2 * blockIdx.x] = __longlong_as_double((long long)(unsigned long long)(mine >> 64));
        partials[2 * blockIdx.x + 1] = __longlong_as_double((long long)(unsigned long long)mine);
        __threadfence();
        s_last = atomicAdd(&sc->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    u128 v = 0;
    for (int q = threadIdx.x; q < (int)gridDim.x; q += blockDim.x)
        v += ((u128)(unsigned long long)__double_as_longlong(__ldcg(partials + 2 * q)) << 64) |
             (unsigned long long)__double_as_longlong(__ldcg(partials + 2 * q + 1));
    v = block_sum_u128(v, red);
    if (threadIdx.x == 0) {
        // the signed 128-bit total, rounded to FP64 once, scaled back by 2^-S
        const long long hi = (long long)(unsigned long long)(v >> 64);
        const unsigned long long lo = (unsigned long long)v;
        const double pap = scale_pow2(fma((double)hi, 18446744073709551616.0, (double)lo), -S);
        sc->ticket = 0;
        sc->next_elem = 0;
        finalize_alpha(sc, pap);
    }
}

}  // namespace nekgb
