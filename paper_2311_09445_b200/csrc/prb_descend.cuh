// The Philox stream and the stratified target: shared by the sample kernels (prb_sample.cu, prb_sample_short.cu).
#pragma once
#include "prb_internal.cuh"
#include "../../include/pearl_prb.h"

#ifdef __CUDACC__

// Philox4x32-10 (Salmon et al., SC'11), first output word only.
__device__ __forceinline__ uint32_t philox4x32_10_word0(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                        uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
        c0 = hi1 ^ c1 ^ k0;
        c1 = lo1;
        c2 = hi0 ^ c3 ^ k1;
        c3 = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c0;
}

// a / b rounded to nearest, from y = 1 / b rounded to nearest: one correction of a y by its exact remainder (P. W. Markstein, "Computation of
// elementary functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34 (1990), theorem 8.3).  The theorem wants a first
// quotient within a unit in the last place; here it is the operands that make the result exact: a has 24 bits (a binary32 sum) and b 11 (strata of a
// cluster), so a / b lies at least 2^-65 of itself from any midpoint of two binary64, and the corrected value is
// within 2^-100 of it before its one rounding.  No overflow or underflow: a is a finite binary32.  Three dependent operations where y is known ahead.
// (tests/test_step_plan.py compares it with the rounded quotient.)
__device__ __forceinline__ double prb_quotient(double a, double b, double y)
{
    const double q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-q, b, a), y, q);
}

// Eq. 1's target of stratum k of B (one draw per equal segment of [0, total), Schaul et al.):
// x_k = (k + u_k) * (total / B) in binary64, two rounded operations, clamped to the binary64 just below
// total; u_k = word 0 of Philox4x32-10(counter = (k, 0, call_lo, call_hi), key = (seed_lo, seed_hi)) * 2^-32.
__device__ __forceinline__ double prb_stratum_target(uint32_t k, uint32_t B, double total, unsigned long long calls, uint64_t seed)
{
    const double seg = __ddiv_rn(total, (double)B);
    const uint32_t r0 = philox4x32_10_word0(k, 0u, (uint32_t)calls, (uint32_t)(calls >> 32), (uint32_t)seed, (uint32_t)(seed >> 32));
    const double u = __dmul_rn((double)r0, 2.3283064365386963e-10);     // * 2^-32, exact
    double x = __dmul_rn(__dadd_rn((double)k, u), seg);
    if (x >= total) x = __longlong_as_double(__double_as_longlong(total) - 1);   // next binary64 below total
    return x;
}

#endif  // __CUDACC__
