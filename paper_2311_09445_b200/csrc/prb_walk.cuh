// One step of the walk from the root to a leaf by a single thread, and the arithmetic of the importance-sampling weights: shared by the
// sample of short rows (prb_sample_short.cu) and the iteration in one kernel (prb_step.cu).
#pragma once
#include "prb_descend.cuh"

#ifdef __CUDACC__

// ---- steps of the walk -----------------------------------------------------------------------------------
// (the child entered is the first whose prefix exceeds the target; a target that has passed every prefix --
// possible by binary32 rounding only -- takes the last positive child and raises CLAMPED)

// Where a step's group of entries lies: a generic address.  (Others: prb_step.cu.)
struct PrbRowAt {
    const float* at;
    __device__ __forceinline__ float4 unit(int q) const { return reinterpret_cast<const float4*>(at)[q]; }
    __device__ __forceinline__ float2 pair() const { return *reinterpret_cast<const float2*>(at); }
    __device__ __forceinline__ float one(uint32_t i) const { return at[i]; }
};

// kWide (many strata per SM): prefixes are compared in binary32 with the largest binary32 not above the target --
// the same answer, and one conversion of the target in place of one per prefix, whose rate bounds the walk there;
// otherwise in binary64, whose conversions are off the chain that bounds a small batch.
template <bool kWide>
struct Target {
    double x;
    float below;
    __device__ __forceinline__ explicit Target(double t) : x(t), below(0.0f) { if (kWide) below = __double2float_rd(t); }
    __device__ __forceinline__ bool past(float prefix) const { return kWide ? prefix <= below : x >= (double)prefix; }
};

// Fanout 2: children c0, c1.
template <bool kWide>
__device__ __forceinline__ bool pick2(double& x, float c0, float c1, unsigned& flags)
{
    const Target<kWide> t(x);
    const bool past0 = t.past(c0), past1 = t.past(__fadd_rn(c0, c1));
    const bool right = past0 && !(past1 && !(c1 > 0.0f));
    if (past1) flags |= (c0 > 0.0f || c1 > 0.0f) ? PEARL_ST_CLAMPED : (PEARL_ST_CLAMPED | PEARL_ST_INTERNAL);
    if (right) x = __dsub_rn(x, (double)c0);
    return right;
}

// Fanout 4.
template <bool kWide>
__device__ __forceinline__ uint32_t pick4(double& x, const float (&c)[4], unsigned& flags)
{
    const float a1 = __fadd_rn(c[0], c[1]), a2 = __fadd_rn(a1, c[2]), a3 = __fadd_rn(a2, c[3]);
    const Target<kWide> t(x);
    uint32_t j = (t.past(c[0]) ? 1u : 0u) + (t.past(a1) ? 1u : 0u) + (t.past(a2) ? 1u : 0u) + (t.past(a3) ? 1u : 0u);
    if (j == 4u) {
        j = c[3] > 0.0f ? 3u : c[2] > 0.0f ? 2u : c[1] > 0.0f ? 1u : 0u;
        flags |= (j > 0u || c[0] > 0.0f) ? PEARL_ST_CLAMPED : (PEARL_ST_CLAMPED | PEARL_ST_INTERNAL);
    }
    if (j > 0u) x = __dsub_rn(x, (double)(j == 1u ? c[0] : j == 2u ? a1 : a2));
    return j;
}

// The 16 entries four levels (fanout 2) or two levels (fanout 4) below a node.
template <int K, bool kWide, typename Row>
__device__ __forceinline__ uint32_t step16(const Row& row, double& x, float& chosen, unsigned& flags)
{
    float e[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 t = row.unit(q);
        e[4 * q] = t.x; e[4 * q + 1] = t.y; e[4 * q + 2] = t.z; e[4 * q + 3] = t.w;
    }
    if constexpr (K == 2) {
        float p8[8], p4[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) p8[i] = __fadd_rn(e[2 * i], e[2 * i + 1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) p4[i] = __fadd_rn(p8[2 * i], p8[2 * i + 1]);
        const bool r0 = pick2<kWide>(x, __fadd_rn(p4[0], p4[1]), __fadd_rn(p4[2], p4[3]), flags);
        const float a0 = r0 ? p4[2] : p4[0], a1 = r0 ? p4[3] : p4[1];
#pragma unroll
        for (int i = 0; i < 4; ++i) p8[i] = r0 ? p8[4 + i] : p8[i];
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = r0 ? e[8 + i] : e[i];
        const bool r1 = pick2<kWide>(x, a0, a1, flags);
        const float b0 = r1 ? p8[2] : p8[0], b1 = r1 ? p8[3] : p8[1];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = r1 ? e[4 + i] : e[i];
        const bool r2 = pick2<kWide>(x, b0, b1, flags);
        const float d0 = r2 ? e[2] : e[0], d1 = r2 ? e[3] : e[1];
        const bool r3 = pick2<kWide>(x, d0, d1, flags);
        chosen = r3 ? d1 : d0;
        return (r0 ? 8u : 0u) + (r1 ? 4u : 0u) + (r2 ? 2u : 0u) + (r3 ? 1u : 0u);
    } else {
        float s[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = __fadd_rn(__fadd_rn(__fadd_rn(e[4 * i], e[4 * i + 1]), e[4 * i + 2]), e[4 * i + 3]);
        const uint32_t j = pick4<kWide>(x, s, flags);
        float c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) c[i] = j == 0u ? e[i] : j == 1u ? e[4 + i] : j == 2u ? e[8 + i] : e[12 + i];
        const uint32_t j2 = pick4<kWide>(x, c, flags);
        chosen = j2 == 0u ? c[0] : j2 == 1u ? c[1] : j2 == 2u ? c[2] : c[3];
        return 4u * j + j2;
    }
}

// One level: the K children of a node.  (From fanout 8 on the chosen child's value is left to the caller, unless kValue.)
template <int K, bool kWide, bool kValue, typename Row>
__device__ __forceinline__ uint32_t step1(const Row& row, double& x, float& chosen, unsigned& flags)
{
    if constexpr (K == 2) {
        const float2 c = row.pair();
        const bool r = pick2<kWide>(x, c.x, c.y, flags);
        chosen = r ? c.y : c.x;
        return r ? 1u : 0u;
    } else if constexpr (K == 4) {
        const float4 t = row.unit(0);
        const float c[4] = { t.x, t.y, t.z, t.w };
        const uint32_t j = pick4<kWide>(x, c, flags);
        chosen = j == 0u ? c[0] : j == 1u ? c[1] : j == 2u ? c[2] : c[3];
        return j;
    } else {
        // prefix <= x, a binary32 against a binary64, is prefix <= (the largest binary32 not above x).
        // All prefixes first (one chain of additions; q[i] lies in front of child i); they do not decrease -- no child is
        // negative -- so the last one passed is found by halving, with selections instead of a comparison for each.
        const float xf = __double2float_rd(x);
        float q[K], e[kValue ? K : 1], all;
        {
            float c[K];
#pragma unroll
            for (int u = 0; u < K / 4; ++u) {
                const float4 t = row.unit(u);
                c[4 * u] = t.x; c[4 * u + 1] = t.y; c[4 * u + 2] = t.z; c[4 * u + 3] = t.w;
            }
            if constexpr (kValue) {
#pragma unroll
                for (int i = 0; i < K; ++i) e[i] = c[i];
            }
            q[0] = 0.0f;
            q[1] = c[0];
#pragma unroll
            for (int i = 2; i < K; ++i) q[i] = __fadd_rn(q[i - 1], c[i - 1]);
            all = __fadd_rn(q[K - 1], c[K - 1]);
        }
        uint32_t j = 0u;
#pragma unroll
        for (int h = K / 2; h > 0; h /= 2) {
            const bool past = q[h] <= xf;
            if (past) j += (uint32_t)h;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                q[i] = past ? q[i + h] : q[i];
                if constexpr (kValue) e[i] = past ? e[i + h] : e[i];
            }
        }
        float before = q[0];
        if constexpr (kValue) chosen = e[0];
        if (all <= xf) {
            flags |= PEARL_ST_CLAMPED;
            j = (uint32_t)K;
            while (j > 0u && !(row.one(j - 1u) > 0.0f)) --j;
            if (j > 0u) --j;
            else flags |= PEARL_ST_INTERNAL;
            before = 0.0f;
#pragma unroll 1
            for (uint32_t i = 0; i < j; ++i) before = i ? __fadd_rn(before, row.one(i)) : row.one(0u);
            if constexpr (kValue) chosen = row.one(j);
        }
        x = __dsub_rn(x, (double)before);              // (0 in front of the first child)
        return j;
    }
}

// ---- weights -----------------------------------------------------------------------------------------------
// n / d for d in [1.7, 2.5], to about a unit in the last place of binary64: a binary32 reciprocal, one Newton step (22 -> 45 bits) and one
// correction of the quotient by its remainder.  Five dependent operations; the general division is a call's worth of them.
__device__ __forceinline__ double quotient_of(double n, double d)
{
    const double y0 = (double)__frcp_rn((float)d);
    const double y = __fma_rn(y0, __fma_rn(-d, y0, 1.0), y0), q = n * y;
    return __fma_rn(__fma_rn(-d, q, n), y, q);
}

// log2 of a positive binary32, in binary64: p = m 2^E with m in (sqrt(1/2), sqrt(2)], t = (m-1)/(m+1),
// ln m = 2 t (1 + t^2/3 + t^4/5 + ...); |t| < 0.172, so the terms left out are below 2^-53 of the sum.
__device__ __forceinline__ double log2_of(float p)
{
    const long long bits = __double_as_longlong((double)p);
    int E = (int)(bits >> 52) - 1023;
    double m = __longlong_as_double((bits & 0x000FFFFFFFFFFFFFll) | 0x3FF0000000000000ll);
    if (m > 1.4142135623730951) { m *= 0.5; E += 1; }
    const double t = quotient_of(m - 1.0, m + 1.0), t2 = t * t, t4 = t2 * t2;
    // (two chains, in t^4: even and odd terms)
    double a = 1.0 / 17.0, b = 1.0 / 19.0;
    a = __fma_rn(a, t4, 1.0 / 13.0); b = __fma_rn(b, t4, 1.0 / 15.0);
    a = __fma_rn(a, t4, 1.0 / 9.0);  b = __fma_rn(b, t4, 1.0 / 11.0);
    a = __fma_rn(a, t4, 1.0 / 5.0);  b = __fma_rn(b, t4, 1.0 / 7.0);
    a = __fma_rn(a, t4, 1.0);        b = __fma_rn(b, t4, 1.0 / 3.0);
    const double S = __fma_rn(b, t2, a);
    return __fma_rn(2.0 * 1.4426950408889634 * t, S, (double)E);
}

// 2^z for z <= 0, rounded to binary32: k = rint(z), 2^z = 2^k e^r with r = (z - k) ln 2 (|r| < 0.35), the
// exponential's series to r^13.  (Below 2^-200 the binary32 is 0 anyway.)
__device__ __forceinline__ float exp2_of(double z)
{
    if (!(z > -200.0)) return 0.0f;
    const double k = rint(z), r = (z - k) * 0.6931471805599453, r2 = r * r;
    double a = 1.0 / 479001600.0, b = 1.0 / 6227020800.0;                                // 1/12!, 1/13!
    a = __fma_rn(a, r2, 1.0 / 3628800.0); b = __fma_rn(b, r2, 1.0 / 39916800.0);
    a = __fma_rn(a, r2, 1.0 / 40320.0);   b = __fma_rn(b, r2, 1.0 / 362880.0);
    a = __fma_rn(a, r2, 1.0 / 720.0);     b = __fma_rn(b, r2, 1.0 / 5040.0);
    a = __fma_rn(a, r2, 1.0 / 24.0);      b = __fma_rn(b, r2, 1.0 / 120.0);
    a = __fma_rn(a, r2, 0.5);             b = __fma_rn(b, r2, 1.0 / 6.0);
    a = __fma_rn(a, r2, 1.0);             b = __fma_rn(b, r2, 1.0);
    const double e = __fma_rn(b, r, a);
    return (float)(e * __longlong_as_double(((long long)k + 1023ll) << 52));
}

#endif  // __CUDACC__
