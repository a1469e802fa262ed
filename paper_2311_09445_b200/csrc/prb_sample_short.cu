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
// memory.  More: a grid; p_min by an atomic per CTA, and no CTA depends on another's being there: one that has copied its rows and does not
// see within some 150 us that all have given theirs leaves its weights to the last that does.  (As a cooperative launch whose CTAs waited for the others it could be no
// programmatic dependent: 4096 strata 24.6 -> 22.6 us a step with its tree kernel, 65536 55.4 -> 53.9.)
#include "prb_walk.cuh"
#include "prb_rows.cuh"

namespace {

constexpr uint32_t kShortThreads = 512;
constexpr uint32_t kShortTopFloats = 5120;           // tree entries staged in shared memory
constexpr uint32_t kMaxSteps = 16;
constexpr uint32_t kMaxCluster = 16;
// Batches of at most this many strata run as one cluster: three warps of strata per CTA.  (The grid form costs a round
// through global memory for the smallest priority.)
constexpr uint32_t kClusterStrata = kPrbClusterStrata;
constexpr uint32_t kMaxSeen = 64;                    // strata warps of a cluster: 8 CTAs x 6 warps, 16 x 3
constexpr uint32_t kGridStrata = 32;                 // strata per CTA of the grid, at least (fewer where rows are long)
constexpr uint32_t kClusterUnits = 1u << 16;         // a cluster copies at most this many units ...
constexpr uint32_t kClusterWords = 400u << 10;       // ... or words
// Looks of a CTA of the grid at whether all have given their smallest priority.  (None in the checked build: there every CTA but the last takes
// the way of those that come too early, which the others hardly ever do.)
#ifdef PEARL_CHECKED
constexpr uint32_t kGridPolls = 0;
#else
constexpr uint32_t kGridPolls = 512;
#endif
constexpr uint32_t kLaneGroupUnits = 160;            // units of a row up to which the lane-group kernel comes next
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
    float* kept;                  // (grid) priorities that wait for their weight: B of them, then a word per CTA
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
        if (many) { if constexpr (K <= 4) j = step16<K, kWide>(PrbRowAt{row}, x, chosen, flags); }
        else j = step1<K, kWide, false>(PrbRowAt{row}, x, chosen, flags);
        if (K > 4) row += j;
        g = (uint32_t)first + j;
    }
    leaf = g;
    p = K > 4 ? *row : chosen;
}

// ---- weights -----------------------------------------------------------------------------------------------
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

// ---- more strata: a grid -------------------------------------------------------------------------------------------
// Every CTA takes a contiguous range of strata, kShortThreads at a time; all its threads copy.  The smallest priority
// is raised (complemented: the word is 0 between calls) with one atomic per CTA, and sample_ticket counts the CTAs that have given
// theirs.  A CTA whose rows are copied forms its weights if all have, or have after a few looks; otherwise it leaves its priorities in `kept`, raises its word there
// and looks once more: either it sees now that all have given theirs, or the last one to do so, which looks for raised words when its own
// rows are copied, finds it (a sequentially consistent fence on either side; both may, and write the same).  So no CTA waits for long, the grid
// need not be co-resident, and the launch is a programmatic dependent like the others.
template <int K, bool kUnits>
__global__ void __launch_bounds__(kShortThreads, 2)
prb_sample_grid_kernel(const __grid_constant__ ShortPlan plan)
{
    __shared__ __align__(16) float s_top[kShortTopFloats];
    __shared__ uint32_t s_idx[kShortThreads];
    __shared__ ShortStep s_step[kMaxSteps];
    __shared__ unsigned s_min, s_flags, s_late;
    __shared__ bool s_all, s_last;
    const uint32_t tid = threadIdx.x, warps = kShortThreads / 32u;
    const uint32_t k_lo = (uint32_t)(((uint64_t)blockIdx.x * plan.B) / gridDim.x);
    const uint32_t k_hi = (uint32_t)(((uint64_t)(blockIdx.x + 1) * plan.B) / gridDim.x);
    const bool exchange = plan.out_w != nullptr && !plan.buffer_norm && !plan.uniform;
    uint32_t* const raised = reinterpret_cast<uint32_t*>(plan.kept + plan.B);      // (a word per CTA)
    StagedUnit unit[kStagedUnits];
#pragma unroll
    for (uint32_t i = 0; i < kStagedUnits; ++i) unit[i] = plan.uniform ? StagedUnit{nullptr, 0u} : staged_unit(plan, s_top, tid + i * kShortThreads);
    if (tid < plan.n_steps) s_step[tid] = plan.step[tid];
    if (tid == 0) { s_min = 0xFFFFFFFFu; s_flags = 0u; s_late = 0u; }
    // (Where a warp's words lie is looked up ahead -- or, at the fanouts whose walks need the registers, behind the walk, where most warps wait anyway: kept across it
    // it was spilled, and every copy read it back.  us a sample in a graph, 262144 slots, 68-byte observations, ahead / behind: fanout 2, 4096 strata 8.99 / 8.18, 65536 17.7 / 15.4;
    // 32, 4096 9.3 / 8.3, 65536 18.3 / 15.5; a step of 16384 27.9 / 26.0 and 24.7 / 23.4; but fanouts 4, 8 and 16, which spill nothing, 24.5 / 24.9, 22.4 / 22.6, 22.4 / 22.8.)
    constexpr bool kBehind = K == 2 || K == 32;
    PrbWordShare share = {};
    if (!kBehind) share = prb_word_share(plan.words, tid >> 5, warps);
    prb_dep_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned long long calls = plan.state->sample_calls;
    const unsigned long long fill = plan.state->fill;
    const float total32 = *plan.level0;
    const bool poisoned = __ldcg(&plan.state->wide_poisoned) != 0u;
    float pmin = 0.0f;
    if (plan.buffer_norm) pmin = plan.min_root ? *plan.min_root : __uint_as_float((unsigned)plan.state->pmin_bits);
    stage(unit);
    if (tid == 0 && exchange) raised[blockIdx.x] = 0u;
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (poisoned) {
        // (CTAs that wait for one another gave up once: see PrbState::wide_poisoned)
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
    const bool kept = k_hi - k_lo > kShortThreads && plan.out_w != nullptr;       // more than one pass: priorities wait for the weight
    float p = 1.0f;
    unsigned flags = 0u, best = 0xFFFFFFFFu, given = 0u;
    for (uint32_t kb = k_lo; kb < k_hi; kb += kShortThreads) {
        const uint32_t n = min(kShortThreads, k_hi - kb), k = kb + tid;
        if (tid < n) {
            const double x = plan.uniform ? 0.0 : prb_stratum_target(k, plan.B, (double)total32, calls, plan.seed);
            const uint32_t leaf = draw<K, true>(plan, s_step, s_top, k, x, calls, fill, p, flags);
            s_idx[tid] = leaf;
            plan.out_idx[k] = (int32_t)leaf;
            best = min(best, __float_as_uint(p));
            if (kept) plan.kept[k] = p;
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
        if (kBehind) share = prb_word_share(plan.words, tid >> 5, warps);
        __syncthreads();
        if (last && tid == kShortThreads - 1u) {
            // this CTA's smallest priority goes out; who else has given one is looked at when the rows have been copied
            if (s_flags) atomicOr(&plan.state->status, s_flags);
            if (exchange) {
                atomicMax(&plan.state->wide_wmax_bits, (unsigned long long)(~s_min));
                asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(given) : "l"(&plan.state->sample_ticket) : "memory");
            }
        }
        gather<kUnits>(plan, share, warps, tid, kb, n, s_idx);
        if (!last) __syncthreads();           // s_idx is rewritten by the next pass
    }
    auto all_given = [&]() {
        uint32_t seen;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&plan.state->sample_ticket) : "memory");
        return seen >= gridDim.x;
    };
    if (exchange) {
        if (tid == kShortThreads - 1u) {
            s_last = given == gridDim.x - 1u;
            // (a while, some 150 us, is waited all the same: CTAs whose SMs other kernels hold start later, and what is left to the last one it does
            // alone.  16384 strata beside matrix products of 4096^3 in bfloat16 on another stream, us a sample and a product, fanout 16: no look 262 and 200, 8 looks
            // 147 and 165, 64 102 and 120, 512 74 and 92; a cooperative launch, whose CTAs all wait, 93 and 93; 2048 strata 61, 21, 25, 31 and 86.  Alone all numbers from 8 on measured
            // the same.)
            bool all = s_last;
            for (uint32_t spins = 0; spins < kGridPolls && !all; ++spins) all = all_given();
            s_all = all;
        }
        __syncthreads();
        if (!s_all) {
            if (!kept && k_lo + tid < k_hi) plan.kept[k_lo + tid] = p;
            __syncthreads();
            if (tid == kShortThreads - 1u) {
                __threadfence();
                atomicExch(raised + blockIdx.x, 1u);
                asm volatile("fence.sc.gpu;" ::: "memory");
                s_all = all_given();
            }
            __syncthreads();
        }
    }
    // (what the last CTA does is the call's tail -- the fence, the looks for raised words and the bookkeeping's atomic each a round trip -- so the fence is
    // another thread's than the read of the minimum, the looks are on their way while the weights are formed, and the atomic does not wait for them: us a
    // sample of 4096 strata in a graph, fanout 8, 262144 slots, one after the other / with an ordinary kernel between them: 8.7 / 9.8 as a cooperative launch, 8.3 / 10.7 with one of
    // these behind the other, 7.65 / 10.1 so; 65536 strata 15.8 / 17.5, 15.0 / 18.2, 14.4 / 17.4)
    if (tid == kShortThreads - 1u) s_min = ~(unsigned)__ldcg(&plan.state->wide_wmax_bits);
    if (tid == 0u && exchange && s_last) asm volatile("fence.sc.gpu;" ::: "memory");
    __syncthreads();
    if (tid == kShortThreads - 1u && prb_ticket(&plan.state->sample_done) == gridDim.x - 1u) {
        // the last CTA to have read what the others have given: the call's bookkeeping
        plan.state->wide_wmax_bits = 0ull;
        plan.state->sample_ticket = 0u;
        plan.state->sample_done = 0u;
        plan.state->sample_calls = calls + 1;
        if (plan.buffer_norm) plan.state->pmin_bits = ~0ull;      // (ready for the next scan)
    }
    uint32_t up = 0u;
    if (exchange && s_last && tid < gridDim.x) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(up) : "l"(raised + tid) : "memory");
    if (exchange) pmin = __uint_as_float(s_min);
    const double log_pmin = plan.uniform ? 0.0 : log2_of(pmin);
    if (plan.out_w != nullptr && (!exchange || s_all))
        for (uint32_t k = k_lo + tid; k < k_hi; k += kShortThreads)
            plan.out_w[k] = plan.uniform ? 1.0f : weight_of(plan, log2_of(kept ? plan.kept[k] : p), log_pmin);
    if (exchange && s_last) {
        // the CTAs that could not wait for this one
        if (up) {
            asm volatile("fence.acq_rel.gpu;" ::: "memory");
            s_idx[atomicAdd(&s_late, 1u)] = tid;
        }
        __syncthreads();
        for (uint32_t e = 0; e < s_late; ++e) {
            const uint32_t c = s_idx[e], hi = (uint32_t)(((uint64_t)(c + 1u) * plan.B) / gridDim.x);
            for (uint32_t k = (uint32_t)(((uint64_t)c * plan.B) / gridDim.x) + tid; k < hi; k += kShortThreads)
                plan.out_w[k] = weight_of(plan, log2_of(__ldcg(plan.kept + k)), log_pmin);
        }
    }
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
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kg, (int)kShortThreads, 0) != cudaSuccess || nb < 1) {
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
    plan.kept = reinterpret_cast<float*>(v.wraw);            // (eight bytes a stratum)
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
        if (grid > kShortThreads) grid = kShortThreads;      // (a thread looks at a CTA's word)
        cfg.gridDim = dim3(grid);
        a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        a[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, short_kernel(v.fanout, true, as_units), plan);
    }
    return e == cudaSuccess ? launches : -1;
}
