// Groups of sibling nodes in registers, and a batch's entries: shared by the kernels of the tree work (prb_tree.cu, prb_step.cu).
#pragma once
#include "prb_internal.cuh"

#ifdef __CUDACC__

constexpr uint32_t kNone = 0xFFFFFFFFu;
template <int K> constexpr uint32_t kLog2 = K == 2 ? 1 : K == 4 ? 2 : K == 8 ? 3 : K == 16 ? 4 : 5;
__host__ __device__ constexpr int ipow(int b, int e) { return e ? b * ipow(b, e - 1) : 1; }

// M entries starting at a multiple of M, from global memory past L1 (other threads of this kernel wrote them).
template <int M>
__device__ __forceinline__ void load_entries(const float* at, float (&e)[M])
{
    if constexpr (M == 2) {
        const float2 t = __ldcg(reinterpret_cast<const float2*>(at));
        e[0] = t.x; e[1] = t.y;
    } else {
#pragma unroll
        for (int q = 0; q < M / 4; ++q) {
            const float4 t = __ldcg(reinterpret_cast<const float4*>(at) + q);
            e[4 * q] = t.x; e[4 * q + 1] = t.y; e[4 * q + 2] = t.z; e[4 * q + 3] = t.w;
        }
    }
}
template <int N, int M>
__device__ __forceinline__ void store_entries(float* at, const float (&e)[M])
{
    if constexpr (N == 1) *at = e[0];
    else if constexpr (N == 2) *reinterpret_cast<float2*>(at) = make_float2(e[0], e[1]);
    else {
#pragma unroll
        for (int q = 0; q < N / 4; ++q) reinterpret_cast<float4*>(at)[q] = make_float4(e[4 * q], e[4 * q + 1], e[4 * q + 2], e[4 * q + 3]);
    }
}
// Left-to-right binary32 sums of groups of K, in place (the first N of e hold the result).
template <int K, int N, int M>
__device__ __forceinline__ void sum_groups(float (&e)[M])
{
#pragma unroll
    for (int j = 0; j < N; ++j) {
        float x = e[j * K];
#pragma unroll
        for (int t = 1; t < K; ++t) x = __fadd_rn(x, e[j * K + t]);
        e[j] = x;
    }
}
// ... and the smallest positive value of groups of K (0 if none).
template <int K, int N, int M>
__device__ __forceinline__ void min_groups(float (&e)[M])
{
#pragma unroll
    for (int j = 0; j < N; ++j) {
        unsigned best = 0xFFFFFFFFu;
#pragma unroll
        for (int t = 0; t < K; ++t) best = min(best, __float_as_uint(e[j * K + t] > 0.0f ? e[j * K + t] : 0.0f) - 1u);
        e[j] = __uint_as_float(best + 1u);
    }
}

// An update entry as read; ok: index in range and not stale.
template <typename Plan>
__device__ __forceinline__ bool entry_ok(const Plan& plan, int32_t i, uint32_t fill, uint32_t cursor, unsigned& flags)
{
    if (i < 0 || (uint32_t)i >= fill) { flags |= PEARL_ST_BAD_INDEX; return false; }
    if (plan.stale | plan.stack) {
        const uint32_t N = plan.capacity, u = (uint32_t)i;
        // one of the `stale` slots written most recently, i.e. overwritten since it was sampled; or one whose
        // history the next insertion overwrites (frames)
        const uint32_t ahead = u >= cursor ? u - cursor : u + N - cursor;       // distance from the cursor along the ring
        if (N - 1u - ahead < plan.stale || ahead < plan.stack) { flags |= PEARL_ST_STALE; return false; }
    }
    return true;
}

// The hash table: linear probing; returns where leaf i lies (the table has twice as many places as entries).
__device__ __forceinline__ uint32_t hash_find(unsigned* key, uint32_t mask, uint32_t shift, uint32_t i)
{
    uint32_t h = prb_hash_place(i, shift);
    while (true) {
        const unsigned old = atomicCAS(key + h, kNone, i);
        if (old == kNone || old == i) return h;
        h = (h + 1u) & mask;
    }
}

#endif  // __CUDACC__
