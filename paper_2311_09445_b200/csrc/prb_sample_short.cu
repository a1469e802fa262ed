// Sampling of short rows (every field below the bulk-copy threshold, one plain transition per slot):
// targets, descents, importance-sampling weights and gather in one launch.
//
// What bounds it is not bandwidth but a chain: state -> top of the tree -> one L2 round trip per step of
// the descent below the staged levels -> rows -> stores, and, across all of it, the smallest priority of the
// batch, which every weight is divided by.  So the kernel is built to keep that chain short.
//
//  * One thread per stratum.  A step reads one contiguous group: the K children of a node, or, for fanouts 2
//    and 4, the 16 descendants four (two) levels down.  A parent is the left-to-right binary32 sum of its
//    children, bit for bit, so the nodes between are re-formed in registers instead of being fetched one
//    level, one round trip, at a time (capacity 10^6, fanout 2: 20 levels in 5 steps, 2 of them in L2).  Only the
//    levels that a step reads are staged in shared memory.
//  * Weights are (p_k / p_min)^-beta with p_min the smallest sampled priority (the power does not increase
//    with p, so this is division by the batch's largest weight), one power per stratum and nothing to
//    normalise afterwards.  p_min is exchanged while the rows are on their way.
//  * Rows are copied word by word, a warp (or a part of one) per row: a lane's word of the row is fixed, so
//    where it lies is looked up once and no index is divided; longer rows unit by unit, by instances of their own (with
//    both copies in one kernel the grid's registers spilled: 65536 rows of 165 bytes 20.6 -> 28.7 us).
//
// Two shapes, by batch size.  Up to kClusterStrata strata: one thread-block cluster of up to 16 CTAs; p_min goes
// through distributed shared memory (each transfer signals the receiver's barrier), nothing through global
// memory.  More: a cooperative grid; p_min by an atomic per CTA, and a CTA waits (bounded) for the others only
// after its rows are copied.
#include "prb_descend.cuh"
#include "prb_rows.cuh"

namespace {

constexpr uint32_t kShortThreads = 512;
constexpr uint32_t kShortTopFloats = 5120;           // tree entries staged in shared memory
constexpr uint32_t kMaxSteps = 16;
constexpr uint32_t kMaxCluster = 16;
// Batches of at most this many strata run as one cluster: three warps of strata per CTA.  (The grid form costs a
// cooperative launch, no programmatic one, and a round through global memory for the smallest priority.)
constexpr uint32_t kClusterStrata = 1536;
constexpr uint32_t kMaxSeen = 64;                    // strata warps of a cluster: 8 CTAs x 6 warps, 16 x 3
constexpr uint32_t kGridStrata = 32;                 // strata per CTA of the cooperative grid, at least (fewer where rows are long)
constexpr uint32_t kClusterUnits = 1u << 16;         // a cluster copies at most this many units ...
constexpr uint32_t kClusterWords = 400u << 10;       // ... or words
constexpr uint32_t kLaneGroupUnits = 160;            // units of a row up to which the lane-group kernel comes next
constexpr uint32_t kShortSpinLimit = 1u << 22;
constexpr uint32_t kNotStaged = 0xFFFFFFFFu;

// One step of the walk: from a node to one of its descendants `levels` levels down.
struct __align__(16) ShortStep {
    uint32_t off;         // level the step reads: entries from level 0's start, in units of 64 (levels start 256-byte aligned)
    uint32_t top;         // where the level lies in the staged copy (entries), or kNotStaged
    uint32_t vec4;        // 16-byte units staged
    uint32_t levels;
};

struct ShortPlan {
    PrbState* state;
    const float* level0;
    const float* min_root;        // the min-tree's root, if the buffer keeps one and the weights want it
    int32_t* out_idx;
    float* out_w;
    uint64_t seed;
    uint32_t B, capacity;
    float beta;
    uint32_t uniform, buffer_norm;
    uint32_t n_steps;
    ShortStep step[kMaxSteps];
    PrbWords words;
#ifdef PEARL_CHECKED
    uint32_t entries[kMaxSteps];  // of the level a step reads, whole 16-entry groups
#endif
};

// ---- steps of the walk -----------------------------------------------------------------------------------
// (the child entered is the first whose prefix exceeds the target; a target that has passed every prefix --
// possible by binary32 rounding only -- takes the last positive child and raises CLAMPED)

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
template <int K, bool kWide>
__device__ __forceinline__ uint32_t step16(const float* row, double& x, float& chosen, unsigned& flags)
{
    float e[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 t = reinterpret_cast<const float4*>(row)[q];
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

// One level: the K children of a node.  (From fanout 8 on the chosen child's value is left to the caller.)
template <int K, bool kWide>
__device__ __forceinline__ uint32_t step1(const float* row, double& x, float& chosen, unsigned& flags)
{
    if constexpr (K == 2) {
        const float2 c = *reinterpret_cast<const float2*>(row);
        const bool r = pick2<kWide>(x, c.x, c.y, flags);
        chosen = r ? c.y : c.x;
        return r ? 1u : 0u;
    } else if constexpr (K == 4) {
        const float4 t = *reinterpret_cast<const float4*>(row);
        const float c[4] = { t.x, t.y, t.z, t.w };
        const uint32_t j = pick4<kWide>(x, c, flags);
        chosen = j == 0u ? c[0] : j == 1u ? c[1] : j == 2u ? c[2] : c[3];
        return j;
    } else {
        // prefix <= x, a binary32 against a binary64, is prefix <= (the largest binary32 not above x).
        // All prefixes first (one chain of additions), then the comparisons as masks, not predicates: counted
        // for the child's number, and the largest prefix passed picked out of them: as signed integers, whose
        // order is that of the values and which put -0.0 (a priority that is accepted; only the prefixes before the
        // first positive child can be it) below every prefix not passed, so that +0.0 is subtracted then.
        const float xf = __double2float_rd(x);
        float r[K];
#pragma unroll
        for (int q = 0; q < K / 4; ++q) {
            const float4 t = reinterpret_cast<const float4*>(row)[q];
            r[4 * q] = t.x; r[4 * q + 1] = t.y; r[4 * q + 2] = t.z; r[4 * q + 3] = t.w;
        }
#pragma unroll
        for (int i = 1; i < K; ++i) r[i] = __fadd_rn(r[i - 1], r[i]);
        uint32_t cnt[K];
        int top[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            asm("set.le.u32.f32 %0, %1, %2;" : "=r"(cnt[i]) : "f"(r[i]), "f"(xf));      // (all ones where passed)
            top[i] = (int)cnt[i] & __float_as_int(r[i]);
        }
#pragma unroll
        for (int h = K / 2; h > 0; h /= 2) {
#pragma unroll
            for (int i = 0; i < h; ++i) { cnt[i] += cnt[i + h]; top[i] = max(top[i], top[i + h]); }
        }
        uint32_t j = 0u - cnt[0];
        int before = top[0];
        if (j == (uint32_t)K) {
            flags |= PEARL_ST_CLAMPED;
            while (j > 0u && !(row[j - 1u] > 0.0f)) --j;
            if (j > 0u) --j;
            else flags |= PEARL_ST_INTERNAL;
            float run = 0.0f;
#pragma unroll 1
            for (uint32_t i = 0; i < j; ++i) run = i ? __fadd_rn(run, row[i]) : row[0];
            before = __float_as_int(run);
        }
        x = __dsub_rn(x, (double)__int_as_float(before));              // (0 in front of the first child)
        return j;
    }
}

template <int K, bool kWide>
__device__ __forceinline__ void walk(const ShortPlan& plan, const ShortStep* steps, const float* s_top, double x, uint32_t& leaf, float& p, unsigned& flags)
{
    constexpr uint32_t lg = K == 2 ? 1u : K == 4 ? 2u : K == 8 ? 3u : K == 16 ? 4u : 5u;
    uint32_t g = 0;
    float chosen = 0.0f;
    ShortStep next = steps[0];
    const float* row = nullptr;
#pragma unroll 1
    for (uint32_t s = 0; s < plan.n_steps; ++s) {
        const ShortStep st = next;
        if (s + 1 < plan.n_steps) next = steps[s + 1];
        const bool many = K <= 4 && st.levels > 1u;
        const uint64_t first = (uint64_t)g << (lg * st.levels);
#ifdef PEARL_CHECKED
        const uint64_t beyond = first + (1ull << (lg * st.levels));
        if (!PRB_IN_BOUNDS(plan, beyond <= plan.entries[s] && (st.top == kNotStaged || st.top + beyond <= kShortTopFloats))) { leaf = 0u; p = 1.0f; return; }
#endif
        // (a generic address: staged level or global memory, one code path)
        row = (st.top != kNotStaged ? s_top + st.top : plan.level0 + ((uint64_t)st.off << 6)) + first;
        uint32_t j;
        if (many) { if constexpr (K <= 4) j = step16<K, kWide>(row, x, chosen, flags); }
        else j = step1<K, kWide>(row, x, chosen, flags);
        if (K > 4) row += j;
        g = (uint32_t)first + j;
    }
    leaf = g;
    p = K > 4 ? *row : chosen;
}

// ---- weights -----------------------------------------------------------------------------------------------
// log2 of a positive binary32, in binary64: p = m 2^E with m in (sqrt(1/2), sqrt(2)], t = (m-1)/(m+1),
// ln m = 2 t (1 + t^2/3 + t^4/5 + ...); |t| < 0.172, so the terms left out are below 2^-53 of the sum.
__device__ __forceinline__ double log2_of(float p)
{
    const long long bits = __double_as_longlong((double)p);
    int E = (int)(bits >> 52) - 1023;
    double m = __longlong_as_double((bits & 0x000FFFFFFFFFFFFFll) | 0x3FF0000000000000ll);
    if (m > 1.4142135623730951) { m *= 0.5; E += 1; }
    const double t = __ddiv_rn(m - 1.0, m + 1.0), t2 = t * t, t4 = t2 * t2;
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

// (p / p_min)^-beta from the two logarithms: 1 where p is the smallest.
// Fewer dependent operations than a general power; against 64-bit references the weights are as close as they
// were with one (the rounding to binary32 is all there is to see).
__device__ __forceinline__ float weight_of(const ShortPlan& plan, double log_p, double log_pmin)
{
    return exp2_of(-(double)plan.beta * (log_p - log_pmin));
}

// Index (and, with uniform replay, all there is to the draw) of stratum k.
template <int K, bool kWide>
__device__ __forceinline__ uint32_t draw(const ShortPlan& plan, const ShortStep* steps, const float* s_top, uint32_t k, double x,
                                         unsigned long long calls, unsigned long long fill, float& p, unsigned& flags)
{
    if (plan.uniform) {
        const uint32_t r0 = philox4x32_10_word0(k, 0u, (uint32_t)calls, (uint32_t)(calls >> 32), (uint32_t)plan.seed, (uint32_t)(plan.seed >> 32));
        return (uint32_t)(((unsigned long long)r0 * fill) >> 32);       // floor(u * fill)
    }
    uint32_t leaf;
    walk<K, kWide>(plan, steps, s_top, x, leaf, p, flags);
    return leaf;
}

// Rows of strata [k0, k0 + n), by `warps` warps; `rank`: this thread's among them.
template <bool kUnits>
__device__ __forceinline__ void gather(const ShortPlan& plan, const PrbWordShare& share, uint32_t warps, uint32_t rank, uint32_t k0, uint32_t n, const uint32_t* s_idx)
{
    auto slot_of = [&](uint32_t r) { return PRB_IN_BOUNDS(plan, s_idx[r] < plan.capacity) ? s_idx[r] : 0u; };
    if constexpr (kUnits) prb_copy_units(plan.words, rank, warps * 32u, k0, n, slot_of);
    else prb_copy_words<false>(plan.words, share, warps, k0, n, slot_of);
}

// What a CTA stages: 16-byte unit `q` of the staged levels, taken one after another (from: nullptr beyond the last).
struct StagedUnit { const float4* from; uint32_t to; };
__device__ __forceinline__ StagedUnit staged_unit(const ShortPlan& plan, const float* s_top, uint32_t q)
{
    StagedUnit o = StagedUnit{nullptr, 0u};
#pragma unroll 1
    for (uint32_t s = 0; s < plan.n_steps; ++s) {
        const ShortStep st = plan.step[s];
        if (st.top == kNotStaged) break;                        // (the staged levels come first)
        if (q < st.vec4) {
            o.from = reinterpret_cast<const float4*>(plan.level0 + ((uint64_t)st.off << 6)) + q;
            o.to = prb_smem_addr(s_top + st.top) + q * 16u;
            break;
        }
        q -= st.vec4;
    }
    return o;
}
constexpr uint32_t kStagedUnits = (kShortTopFloats / 4u + kShortThreads - 1u) / kShortThreads;      // per thread
__device__ __forceinline__ void stage(const StagedUnit (&u)[kStagedUnits])
{
#pragma unroll
    for (uint32_t i = 0; i < kStagedUnits; ++i)
        if (u[i].from != nullptr) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(u[i].to), "l"(u[i].from) : "memory");
}

// ---- up to kClusterStrata strata: one cluster -----------------------------------------------------------------
// The first warps of a CTA hold its strata, a thread each, and look after the weights; the others copy the rows
// as soon as the indices are known (all do both where that would leave fewer than half of them to copy).
// Launched as a programmatic dependent: until the wait the kernel before it may still be running, nothing is read or
// written, and all that depends on the arguments alone is done -- where every thread's words and staged units
// lie, and a dry run of the arithmetic, which fetches its constants (the first use of a binary64 constant was
// measured at 430 cycles, each further line of them at 84).
// From that wait to the last store, fanout 16, 2^20 slots, 64 strata: 7000 cycles; the kernel before it (a lane group
// per stratum over 32 CTAs, raw weights through global memory and a ticket, rows field by field) took 16000, 5400 of
// them the last CTA's division.  CTAs: 2, 4, 8 or 16 strata each measured the same within 1 %; 4.
struct __align__(16) SmallestSeen { double log_p; unsigned long long p_bits; };

template <int K, bool kUnits>
__global__ void __launch_bounds__(kShortThreads, K == 32 ? 1 : 2)
prb_sample_cluster_kernel(const __grid_constant__ ShortPlan plan)
{
    __shared__ __align__(16) float s_top[kShortTopFloats];
    __shared__ uint32_t s_idx[kShortThreads];
    __shared__ ShortStep s_step[kMaxSteps];
    __shared__ SmallestSeen s_seen[kMaxSeen];                  // the smallest sampled priority of every strata warp of the cluster
    __shared__ __align__(8) unsigned long long s_bar;          // completes when all of them are there
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, warps = blockDim.x >> 5;
    const uint32_t k_lo = (uint32_t)(((uint64_t)blockIdx.x * plan.B) / gridDim.x);
    const uint32_t k_hi = (uint32_t)(((uint64_t)(blockIdx.x + 1) * plan.B) / gridDim.x);
    const uint32_t n = k_hi - k_lo, k = k_lo + tid;
    const bool mine = tid < n;
    const uint32_t strata_warps = ((plan.B + gridDim.x - 1) / gridDim.x + 31u) / 32u;      // the same in every CTA
    const bool split = strata_warps * 2u <= warps;
    const uint32_t first_copier = split ? strata_warps : 0u;
    const bool copies = warp >= first_copier;
    const uint32_t bar = prb_smem_addr(&s_bar);
    if (tid < plan.n_steps) s_step[tid] = plan.step[tid];
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)sizeof(SmallestSeen) * gridDim.x * strata_warps) : "memory");
    }
    PrbWordShare share = {};
    if (copies) share = prb_word_share(plan.words, warp - first_copier, warps - first_copier);
    StagedUnit unit[kStagedUnits];
#pragma unroll
    for (uint32_t i = 0; i < kStagedUnits; ++i) unit[i] = plan.uniform ? StagedUnit{nullptr, 0u} : staged_unit(plan, s_top, tid + i * blockDim.x);
    if (warp < strata_warps) {
        const double dry = prb_stratum_target(k, plan.B, 1.0 + (double)tid, 0ull, plan.seed);
        if (weight_of(plan, log2_of(2.0f + (float)dry), 1.0) > 1.5f) s_idx[tid] = 0u;          // (never: 2^-x for x >= 0)
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // (every CTA's s_bar can be signalled)
    prb_dep_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned long long calls = plan.state->sample_calls;
    const unsigned long long fill = plan.state->fill;
    const float total32 = *plan.level0;
    float pmin = 0.0f;
    if (plan.buffer_norm) pmin = plan.min_root ? *plan.min_root : __uint_as_float((unsigned)plan.state->pmin_bits);
    stage(unit);
    if (fill == 0 || (!plan.uniform && !(total32 > 0.0f))) {
        // an empty buffer: nothing is written (every CTA sees the same)
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (blockIdx.x == 0 && tid == 0) {
            atomicOr(&plan.state->status, PEARL_ST_EMPTY);
            if (plan.buffer_norm) plan.state->pmin_bits = ~0ull;
        }
        return;
    }
    double x = 0.0;
    if (mine) x = prb_stratum_target(k, plan.B, (double)total32, calls, plan.seed);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();                                           // the staged levels are in place
    float p = 1.0f;
    uint32_t leaf = 0;
    if (warp < strata_warps) {
        unsigned flags = 0u;
        if (mine) { leaf = draw<K, false>(plan, s_step, s_top, k, x, calls, fill, p, flags); s_idx[tid] = leaf; }
        __syncwarp();
        if (split) asm volatile("bar.arrive 1, %0;" ::"r"(blockDim.x) : "memory");      // the copying warps may go on
        if (flags) atomicOr(&plan.state->status, flags);
    }
    if (copies) {
        asm volatile("bar.sync 1, %0;" ::"r"(blockDim.x) : "memory");
        if (split) { gather<kUnits>(plan, share, warps - first_copier, tid - first_copier * 32u, k_lo, n, s_idx); return; }
    }
    double log_p = 0.0;
    if (warp < strata_warps) {
        // the warp's smallest priority and its logarithm go to every CTA of the cluster; a transfer signals the
        // receiver's barrier  (priorities are not negative: they order like their bits)
        log_p = log2_of(p);
        const unsigned bits = mine ? __float_as_uint(p) : 0x7F800000u;
        const unsigned least = __reduce_min_sync(0xFFFFFFFFu, bits);
        const double log_least = __shfl_sync(0xFFFFFFFFu, log_p, __ffs(__ballot_sync(0xFFFFFFFFu, bits == least)) - 1);
        if (lane < gridDim.x) {
            uint32_t to, to_bar;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(prb_smem_addr(s_seen + blockIdx.x * strata_warps + warp)), "r"(lane));
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to_bar) : "r"(bar), "r"(lane));
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];"
                         ::"r"(to), "l"(__double_as_longlong(log_least)), "l"((unsigned long long)least), "r"(to_bar) : "memory");
        }
        if (mine) plan.out_idx[k] = (int32_t)leaf;
    }
    if (!split) gather<kUnits>(plan, share, warps, tid, k_lo, n, s_idx);
    // (the first warp always gets here: it keeps the CTA's shared memory until every value has come)
    if (warp >= strata_warps) return;
    if (prb_wait_first_phase<true>(plan.state, bar) == kPrbNever) return;
    if (blockIdx.x == 0 && tid == 0) {
        plan.state->sample_calls = calls + 1;                  // (every CTA has drawn)
        if (plan.buffer_norm) plan.state->pmin_bits = ~0ull;   // (ready for the next scan)
    }
    if (plan.out_w == nullptr) return;
    __syncwarp();
    double log_pmin;
    if (plan.buffer_norm) {
        log_pmin = log2_of(pmin);
    } else {
        unsigned best = 0xFFFFFFFFu;
        double log_best = 0.0;
        for (uint32_t i = lane; i < gridDim.x * strata_warps; i += 32u) {
            const unsigned b = (unsigned)s_seen[i].p_bits;
            if (b < best) { best = b; log_best = s_seen[i].log_p; }
        }
        __syncwarp();
        const unsigned least = __reduce_min_sync(0xFFFFFFFFu, best);
        log_pmin = __shfl_sync(0xFFFFFFFFu, log_best, __ffs(__ballot_sync(0xFFFFFFFFu, best == least)) - 1);
    }
    if (mine) plan.out_w[k] = plan.uniform ? 1.0f : weight_of(plan, log_p, log_pmin);
}

// ---- more strata: a cooperative grid ---------------------------------------------------------------------------
// Every CTA takes a contiguous range of strata, kShortThreads at a time; all its threads copy.  The smallest priority
// is raised (complemented: the word is 0 between calls) with one atomic per CTA, and sample_ticket counts the
// CTAs that have given theirs, then those that have read the answer.
template <int K, bool kUnits>
__global__ void __launch_bounds__(kShortThreads, 2)
prb_sample_grid_kernel(const __grid_constant__ ShortPlan plan)
{
    __shared__ __align__(16) float s_top[kShortTopFloats];
    __shared__ uint32_t s_idx[kShortThreads];
    __shared__ ShortStep s_step[kMaxSteps];
    __shared__ unsigned s_min, s_flags;
    __shared__ int s_ok;
    const uint32_t tid = threadIdx.x, warps = kShortThreads / 32u;
    const uint32_t k_lo = (uint32_t)(((uint64_t)blockIdx.x * plan.B) / gridDim.x);
    const uint32_t k_hi = (uint32_t)(((uint64_t)(blockIdx.x + 1) * plan.B) / gridDim.x);
    const unsigned long long calls = plan.state->sample_calls;
    const unsigned long long fill = plan.state->fill;
    const float total32 = *plan.level0;
    const bool poisoned = __ldcg(&plan.state->wide_poisoned) != 0u;
    float pmin = 0.0f;
    if (plan.buffer_norm) pmin = plan.min_root ? *plan.min_root : __uint_as_float((unsigned)plan.state->pmin_bits);
    if (!plan.uniform) {
        StagedUnit unit[kStagedUnits];
#pragma unroll
        for (uint32_t i = 0; i < kStagedUnits; ++i) unit[i] = staged_unit(plan, s_top, tid + i * kShortThreads);
        stage(unit);
    }
    if (tid < plan.n_steps) s_step[tid] = plan.step[tid];
    if (tid == 0) { s_min = 0xFFFFFFFFu; s_flags = 0u; }
    const PrbWordShare share = prb_word_share(plan.words, tid >> 5, warps);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (poisoned) {
        // (a launch of co-resident CTAs gave up at its barrier once: see PrbState::wide_poisoned)
        if (tid == 0 && blockIdx.x == 0) atomicOr(&plan.state->status, PEARL_ST_INTERNAL);
        return;
    }
    if (fill == 0 || (!plan.uniform && !(total32 > 0.0f))) {
        if (blockIdx.x == 0 && tid == 0) {
            atomicOr(&plan.state->status, PEARL_ST_EMPTY);
            if (plan.buffer_norm) plan.state->pmin_bits = ~0ull;
        }
        return;
    }
    const bool exchange = plan.out_w != nullptr && !plan.buffer_norm && !plan.uniform;
    const bool kept = k_hi - k_lo > kShortThreads && plan.out_w != nullptr;       // more than one pass: priorities wait in out_w for the weight
    float p = 1.0f;
    unsigned flags = 0u, best = 0xFFFFFFFFu;
    for (uint32_t kb = k_lo; kb < k_hi; kb += kShortThreads) {
        const uint32_t n = min(kShortThreads, k_hi - kb), k = kb + tid;
        if (tid < n) {
            const double x = plan.uniform ? 0.0 : prb_stratum_target(k, plan.B, (double)total32, calls, plan.seed);
            const uint32_t leaf = draw<K, true>(plan, s_step, s_top, k, x, calls, fill, p, flags);
            s_idx[tid] = leaf;
            plan.out_idx[k] = (int32_t)leaf;
            best = min(best, __float_as_uint(p));
            if (kept) plan.out_w[k] = p;
        }
        const bool last = kb + kShortThreads >= k_hi;
        __syncwarp();
        if (last) {
            const unsigned b = __reduce_min_sync(0xFFFFFFFFu, best);
            const unsigned fl = __reduce_or_sync(0xFFFFFFFFu, flags);
            if ((tid & 31u) == 0u) {
                if (b != 0xFFFFFFFFu) atomicMin(&s_min, b);
                if (fl) atomicOr(&s_flags, fl);
            }
        }
        __syncthreads();
        if (last && tid == kShortThreads - 1u) {
            // this CTA's smallest priority goes out; the answer is looked at when the rows have been copied
            if (s_flags) atomicOr(&plan.state->status, s_flags);
            if (exchange) atomicMax(&plan.state->wide_wmax_bits, (unsigned long long)(~s_min));
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&plan.state->sample_ticket) : "memory");
        }
        gather<kUnits>(plan, share, warps, tid, kb, n, s_idx);
        if (!last) __syncthreads();           // s_idx is rewritten by the next pass
    }
    if (tid == kShortThreads - 1u) {
        // (bounded wait; the grid is co-resident)
        int ok = 0;
        for (uint32_t spins = 0; spins < kShortSpinLimit && !ok; ++spins) {
            uint32_t seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&plan.state->sample_ticket) : "memory");
            ok = seen >= gridDim.x;
        }
        s_ok = ok;
        s_min = ~(unsigned)__ldcg(&plan.state->wide_wmax_bits);
        if (!ok) { atomicOr(&plan.state->status, PEARL_ST_INTERNAL); atomicExch(&plan.state->wide_poisoned, 1u); }
        else if (prb_ticket(&plan.state->sample_ticket) == 2u * gridDim.x - 1u) {
            // the last CTA to have read the minimum: the call's bookkeeping
            plan.state->wide_wmax_bits = 0ull;
            plan.state->sample_ticket = 0u;
            plan.state->sample_calls = calls + 1;
            if (plan.buffer_norm) plan.state->pmin_bits = ~0ull;      // (ready for the next scan)
        }
    }
    __syncthreads();
    if (!s_ok || plan.out_w == nullptr) return;
    if (exchange) pmin = __uint_as_float(s_min);
    const double log_pmin = plan.uniform ? 0.0 : log2_of(pmin);
    for (uint32_t k = k_lo + tid; k < k_hi; k += kShortThreads)
        plan.out_w[k] = plan.uniform ? 1.0f : weight_of(plan, log2_of(kept ? plan.out_w[k] : p), log_pmin);
}

using ShortKernel = void (*)(ShortPlan);
template <int K>
ShortKernel short_kernel_k(bool grid, bool units)
{
    if (grid) return units ? prb_sample_grid_kernel<K, true> : prb_sample_grid_kernel<K, false>;
    return units ? prb_sample_cluster_kernel<K, true> : prb_sample_cluster_kernel<K, false>;
}
ShortKernel short_kernel(uint32_t fanout, bool grid, bool units)
{
    switch (fanout) {
    case 2: return short_kernel_k<2>(grid, units);
    case 4: return short_kernel_k<4>(grid, units);
    case 8: return short_kernel_k<8>(grid, units);
    case 16: return short_kernel_k<16>(grid, units);
    default: return short_kernel_k<32>(grid, units);
    }
}

// What this device runs: CTAs a cluster may have (16 needs the opt-in and an SM group that holds it), and
// co-resident CTAs of the grid form per SM.
struct ShortLimits { uint32_t cluster, per_sm; };
const ShortLimits* short_limits(uint32_t fanout, int ki, int dev, bool units)
{
    static ShortLimits cache[kPrbMaxDevices][6][2];
    ShortLimits& l = cache[dev][ki][units ? 1 : 0];
    if (l.cluster) return &l;
    ShortKernel kc = short_kernel(fanout, false, units), kg = short_kernel(fanout, true, units);
    uint32_t cluster = 8;
    if (cudaFuncSetAttribute(kc, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kMaxCluster);
        cfg.blockDim = dim3(kShortThreads);
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = kMaxCluster; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a;
        cfg.numAttrs = 1;
        int fits = 0;
        if (cudaOccupancyMaxActiveClusters(&fits, kc, &cfg) == cudaSuccess && fits >= 1) cluster = kMaxCluster;
    }
    cudaGetLastError();
    int nb = 0, coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kg, (int)kShortThreads, 0) != cudaSuccess || nb < 1) {
        cudaGetLastError();
        nb = 0;                                          // (no grid form here)
    }
    l.per_sm = nb > 2 ? 2u : (uint32_t)nb;
    l.cluster = cluster;
    return &l;
}

}  // namespace

int prb_launch_sample_short(const PrbView& v, uint32_t B, float beta, uint64_t seed, int32_t* d_idx, float* d_w, const PrbBatch& dst,
                            cudaStream_t s, int uniform, int buffer_norm)
{
    const int dev = prb_current_device();
    ShortPlan plan;
    plan.words = prb_plan_words(v, dst);
    const PrbWords& rows = plan.words;
    // Which kernel.  The cluster's 16 SMs while they have little to copy: up to kClusterUnits units (kClusterWords words where a
    // row's granules are small).  Beyond, up to kClusterStrata strata: rows of medium length go to the lane-group kernel
    // (prb_sample.cu: every SM copies, and no grid-wide minimum); longer ones, and more strata, to the grid, with fewer
    // strata to a CTA where rows are long.  us a call, cluster / lane groups / grid, fanout 16: 512 rows of 1 KB 6.6 / 6.9 /
    // 8.6, 1024 of 1 KB 8.7 / 8.4 / 9.3, 512 of 2 KB 7.7 / 7.0 / 8.5, 1024 of 2 KB 11.5 / 8.3 / 9.0; 256 of 4 KB 8.1 / 9.3 / 8.5,
    // 512 of 4 KB 11.5 / 9.6 / 9.1, 256 of 14 KB 17 / 21 / 10.7, 1024 of 14 KB 57 / 22 / 13.5.
    const bool longer = rows.n_words > kPrbMostWords;
    const uint64_t units = (uint64_t)B * rows.units, words = (uint64_t)B * rows.n_words;
    const bool cluster = B <= kClusterStrata && (!longer || rows.units == 0u || (rows.fine ? words <= kClusterWords : units <= kClusterUnits));
    if (!cluster && B <= kClusterStrata && !rows.fine && rows.units <= kLaneGroupUnits) return 0;
    const bool as_units = rows.units != 0u && longer && (!cluster || !rows.fine);
    const ShortLimits* lim = short_limits(v.fanout, (int)v.log2_fanout, dev, as_units);
    if (!cluster && lim->per_sm == 0) return 0;
    plan.state = v.state;
    plan.level0 = v.level[0];
    plan.out_idx = d_idx;
    plan.out_w = d_w;
    plan.seed = seed;
    plan.B = B;
    plan.capacity = (uint32_t)v.capacity;
    plan.beta = beta;
    plan.uniform = uniform ? 1u : 0u;
    plan.buffer_norm = (buffer_norm && !uniform) ? 1u : 0u;
    plan.min_root = (plan.buffer_norm && v.min_off) ? v.level[0] + v.min_off : nullptr;
    // the walk: single levels first until what is left is a whole number of 16-entry steps (fanouts 2 and 4)
    const uint32_t per = v.fanout == 2 ? 4u : v.fanout == 4 ? 2u : 1u;
    uint32_t n = 0, at = 0;
    bool staging = true;
    for (uint32_t l = 0; l < v.depth;) {
        const uint32_t h = (v.depth - l) % per ? 1u : per;
        l += h;
        if (n == kMaxSteps) return -1;
        ShortStep& st = plan.step[n++];
        st.off = (uint32_t)((uint64_t)(v.level[l] - v.level[0]) >> 6);
        st.levels = h;
        // whole 16-entry groups (a level's end is padded with zeros to a 256-byte boundary)
        const uint32_t entries = (v.level_alloc[l] + 15u) / 16u * 16u;
#ifdef PEARL_CHECKED
        plan.entries[n - 1] = entries;
#endif
        staging = staging && entries <= kShortTopFloats && at + entries <= kShortTopFloats;
        st.top = staging ? at : kNotStaged;
        st.vec4 = staging ? entries / 4u : 0u;
        if (staging) at += entries;
    }
    plan.n_steps = n;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cudaLaunchAttribute a[2];
    cfg.attrs = a;
    int launches = 1;
    if (plan.buffer_norm && v.min_off == 0) {
        // no min-tree to read the smallest priority from: the scan of the leaves goes first
        if (prb_launch_leaf_min(v, s) < 0) return -1;
        launches = 2;
    }
    cudaError_t e;
    cfg.blockDim = dim3(kShortThreads);
    if (cluster) {
        // a few strata per CTA (their rows are copied by all its warps), up to the whole cluster
        uint32_t ctas = 1;
        while (ctas < lim->cluster && ctas * 4u < B) ctas *= 2u;
        cfg.gridDim = dim3(ctas);
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = ctas; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        a[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        a[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.numAttrs = 2;
        e = cudaLaunchKernelEx(&cfg, short_kernel(v.fanout, false, as_units), plan);
    } else {
        const uint32_t strata = !as_units ? kGridStrata : rows.units >= 4000u ? 1u : rows.units >= 400u ? 4u : rows.units >= 100u ? 8u : kGridStrata;
        uint32_t grid = (B + strata - 1) / strata;
        const uint32_t room = (uint32_t)prb_sm_count() * lim->per_sm;
        if (grid > room) grid = room;
        cfg.gridDim = dim3(grid);
        a[0].id = cudaLaunchAttributeCooperative;
        a[0].val.cooperative = 1;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, short_kernel(v.fanout, true, as_units), plan);
    }
    return e == cudaSuccess ? launches : -1;
}
