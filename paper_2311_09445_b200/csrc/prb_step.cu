// An iteration of short rows -- priority update, insertion, and the sample of the next batch -- in one launch, and the same
// tree work without the sample: one thread-block cluster.
//
// What bounds it is a chain, and this file is about its length: inputs -> transform -> leaves -> the levels above them ->
// the root -> targets -> descents -> rows.  As two kernels (prb_tree.cu, then prb_sample_short.cu) every pass over a level
// below the staged top was a round trip through L2 and a half, the staged top was re-summed by one CTA, and the sample
// read all of it again behind a kernel boundary.  Here
//  * the tree is cut at level U (at most kMostUpper nodes).  What lies below a node of level U belongs to one CTA (nodes
//    dealt round-robin): it alone writes there, and no other CTA has to be waited for below level U;
//  * levels go in steps of a group of 8, 16 or 32 entries (fanouts 2 and 4: four and two levels a step).  The CTA stages
//    the levels of the first steps below U whole, as far as that pays (kPortionFloats); of the steps below those it fetches
//    the groups that its entries fall into, all of them at once and as soon as the indices are known -- while the transform
//    runs -- into rows of shared memory, which a hash table per step finds.  New values are written into the rows and summed up
//    from row to row, from staged level to staged level: what separates the steps is a barrier of eight warps, not
//    a round trip;
//  * level U goes from every CTA to every CTA through distributed shared memory (each transfer signals the receiver's barrier; so does an
//    arrival that releases the staged levels), and every CTA sums up the few levels above it;
//  * a descent walks those in its own shared memory, the staged levels in their owners' (distributed shared memory), and only the
//    last steps in L2, where a fence off the chain has made them visible;
//  * rows of the insertion are copied by warps of their own meanwhile, and a sampled slot that this very call inserts is
//    read from the insertion's batch: nobody waits for the copy.
// us a step, two kernels / this one: captured, fanout 16, 2^20 slots, 256 + 256 entries 10.0 / 8.3; fanout 2, 10^6 slots, 1000 + 777
// 14.9 / 12.6; called eagerly, 32 entries of a 4096-slot binary tree 10.2 / 7.5, 64 + 64 of 2^20 slots 11.8 / 8.8; through pinned host
// arrays, 256 + 256 entries, fanout 16, 2^20 slots 37.7 / 36.4, fanout 2, 2^17 slots 39.6 / 36.1.  Of the 8.3: 1.4 between the kernels, 1.4 until the groups are there, 1.2 up to level U, 0.7 to
// the root, 2.1 down to the leaf, 1.2 for weights and rows.
#include "prb_walk.cuh"
#include "prb_groups.cuh"
#include "prb_rows.cuh"
#include "prb_tree.cuh"

namespace {

// Warps: 8 that do the tree work and hold the strata, 8 that look after the entries and copy rows, and for a small batch two more that have the
// insertion's groups of leaves, which all fall to one CTA or two (by the other warps, one after another: 1000 cycles of a chain of 13500).
constexpr uint32_t kTreeWarps = 8, kTreeThreads = 256, kCopyThreads = 256;
template <uint32_t kEach> constexpr uint32_t kGroupThreads = kEach == 1u ? 64u : 0u;
template <uint32_t kEach> constexpr uint32_t kStepThreads = kTreeThreads + kCopyThreads + kGroupThreads<kEach>;
constexpr uint32_t kStepParts = 16;                         // CTAs of the cluster, at most
constexpr uint32_t kMostEach = 4;                           // entries of the batch a thread looks at, at most
constexpr uint32_t kMostEntries = kTreeThreads * kMostEach; // update entries, and inserted leaves
// Nodes of level U; half of it but for fanout 32, whose next cut would be 32 times coarser.  (Up to 1024 for all: fanout 16, 2^18 slots, steps of 256 + 256 7.02 -> 7.35 us,
// fanout 4 9.20 -> 9.59, fanout 2, 2^14 slots 7.00 -> 7.34.)
constexpr uint32_t kMostUpper = 1024;
constexpr uint32_t kUpperLevels = 12;
// Staged entries below level U, per CTA: of a batch of one entry a thread, and of larger ones.  All of them are fetched and every staged group is looked
// at whatever the batch, so a small batch rather works one more level off as groups of its own: us a call in a graph, 14336 / 8192: fanout 8, 2^20 slots, updates
// of 32 5.67 / 4.08 (4.88 with prb_tree.cu), steps of 32 8.81 / 7.42; 2^23 slots 5.81 / 4.63; fanout 16, 2^21 slots 4.91 / 4.05, steps of 256 + 256
// 8.79 / 8.20; fanout 32, 2^22 slots 4.75 / 3.99.  400 + 400 entries in the same trees: fanout 8 9.56 / 9.20, but 16 9.04 / 9.32, 32 9.19 / 9.58, 4 11.74 / 12.00.
constexpr uint32_t kPortionFloats = 8192, kPortionFloatsMany = 14336;
constexpr uint32_t kMostStaged = 4, kMostPasses = 8;
constexpr uint32_t kMostSeen = 64;
constexpr uint32_t kStepSmem = 200u * 1024u;

template <int K> constexpr int kSpan = K == 2 ? 4 : K == 4 ? 2 : 1;                     // levels of a step
template <int K> constexpr int kGroup = ipow(K, kSpan<K>);                              // entries of a group
template <int K> constexpr uint32_t kLogGroup = kLog2<K> * (uint32_t)kSpan<K>;

struct StepPlan {
    PrbState* state;
    float* level0;
    const int32_t* idx;
    const float* val;
    const float* prio;
    const unsigned char* done;
    int32_t* out_idx;
    float* out_w;
    uint64_t seed, min_off;
    uint32_t capacity, depth, B_upd, n, B;
    float alpha, eps, beta;
    uint32_t raw, stale, stack;
    uint32_t moves_rows;                      // the insertion's rows are this kernel's
    uint32_t linked;                          // the inputs lie in mapped host memory
    uint32_t U, staged, passes;               // cut, staged steps below it, steps below those
    uint32_t n_u, own, own4;                  // nodes of level U; of them a CTA's, at most, and in units of four
    uint32_t log_parts;
    uint32_t rows, list;                      // groups held at a time (per step); entries: positions of the batch, or capacity of the list
    uint32_t portion_units, portion_floats;
    uint32_t leaf_mask, leaf_shift, node_mask, node_shift;       // hash tables: places less one, 32 - log2 of the places
    uint32_t up_floats;
    // byte offsets in dynamic shared memory
    uint32_t o_own, o_portion, o_dirty, dirty_bytes, o_rows, o_nodes, o_place, o_leaf, o_list;
    uint32_t off[PRB_MAX_LEVELS];             // level l starts off[l] * 64 entries behind level 0
    uint32_t up[kUpperLevels];                // level l <= U in the upper levels' copy (entries)
    uint32_t portion_at[kMostStaged + 1];     // staged step s (1 ..) in the portion (entries)
    uint32_t dirty_at[kMostStaged + 1];
    PrbWords in, out;
};

// Groups held in shared memory lie 16 bytes apart, so that threads that read a group each do not meet in a bank.
template <int K> constexpr uint32_t kPitch = (uint32_t)kGroup<K> + 4u;
// ... entry f of a staged level's part
template <int K> __device__ __forceinline__ uint32_t padded(uint32_t f) { return (f >> kLogGroup<K>) * kPitch<K> + (f & (uint32_t)(kGroup<K> - 1)); }

// Barriers: 1 the tree warps' own (8 with the insertion's groups), 4 the other warps'; 7 the list of entries, 5 their groups are there; 6 the
// groups are done with; 3 everything below level U is stored; 2 the sampled indices are there.
__device__ __forceinline__ void tree_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kTreeThreads) : "memory"); }
// ... which says whether all its threads still hold sound sums
__device__ __forceinline__ bool tree_sync_all(bool sound)
{
    uint32_t all;
    asm volatile("{ .reg .pred p, q; setp.ne.u32 p, %1, 0; barrier.cta.red.and.pred q, 1, %2, p; selp.u32 %0, 1, 0, q; }" : "=r"(all) : "r"(sound ? 1u : 0u), "n"(kTreeThreads) : "memory");
    return all != 0u;
}
template <uint32_t kEach> __device__ __forceinline__ void sum_sync() { asm volatile("bar.sync 8, %0;" ::"n"(kTreeThreads + kGroupThreads<kEach>) : "memory"); }
template <uint32_t kEach> __device__ __forceinline__ void copy_sync() { asm volatile("bar.sync 4, %0;" ::"n"(kCopyThreads + kGroupThreads<kEach>) : "memory"); }

struct StepCtx {
    const StepPlan& plan;
    const uint32_t* off;
    __device__ __forceinline__ float* level(uint32_t l) const { return plan.level0 + ((uint64_t)off[l] << 6); }
};

// The levels between a group of level `child` and its node a, kSpan levels up, and that node: summed up in registers and stored.
// (kLeast: the min-tree's nodes, min_off behind the sum tree's)
template <int K, bool kLeast, int S>
__device__ __forceinline__ void sum_up(const StepCtx& c, uint64_t min_off, uint32_t child, uint32_t a, float (&e)[kGroup<K>])
{
    if constexpr (S < kSpan<K>) {
        constexpr int N = ipow(K, kSpan<K> - 1 - S);
        if constexpr (kLeast) min_groups<K, N>(e);
        else sum_groups<K, N>(e);
        store_entries<N>(c.level(child - 1 - S) + min_off + (uint64_t)a * N, e);
        sum_up<K, kLeast, S + 1>(c, min_off, child, a, e);
    }
}
template <int M>
__device__ __forceinline__ void load_group(const float* from, float (&e)[M])
{
#pragma unroll
    for (int q = 0; q < M / 4; ++q) {
        const float4 t = reinterpret_cast<const float4*>(from)[q];
        e[4 * q] = t.x; e[4 * q + 1] = t.y; e[4 * q + 2] = t.z; e[4 * q + 3] = t.w;
    }
}

// Upper levels: node i of level l - H and what lies between, from the entries of level l (which starts at `at`) under it.
template <int K, bool kLeast, int H, int S>
__device__ __forceinline__ void sum_up_top(const StepCtx& c, float* up, uint64_t min_off, bool store, uint32_t l, uint32_t i, float (&e)[ipow(K, H)])
{
    if constexpr (S < H) {
        constexpr int N = ipow(K, H - 1 - S);
        if constexpr (kLeast) min_groups<K, N>(e);
        else sum_groups<K, N>(e);
        store_entries<N>(up + c.plan.up[l - 1 - S] + i * N, e);
        if (store) store_entries<N>(c.level(l - 1 - S) + min_off + (uint64_t)i * N, e);
        sum_up_top<K, kLeast, H, S + 1>(c, up, min_off, store, l, i, e);
    }
}
template <int K, bool kLeast, int H>
__device__ __forceinline__ void top_group(const StepCtx& c, float* up, uint64_t min_off, bool store, uint32_t l, uint32_t at, uint32_t i)
{
    constexpr int M = ipow(K, H);
    float e[M];
    if (!PRB_IN_BOUNDS(c.plan, at + (i + 1u) * M <= c.plan.up_floats)) return;
    const float* const from = up + at + i * M;
    if constexpr (M == 2) {
        const float2 t = *reinterpret_cast<const float2*>(from);
        e[0] = t.x; e[1] = t.y;
    } else {
        load_group<M>(from, e);
    }
    sum_up_top<K, kLeast, H, 0>(c, up, min_off, store, l, i, e);
}

// Rows of the walk: a group in a peer's portion, a group in L2.
struct RowOfPeer {
    uint32_t at;
    __device__ __forceinline__ float4 unit(int q) const
    {
        float4 t;
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(at + (uint32_t)q * 16u) : "memory");
        return t;
    }
    __device__ __forceinline__ float one(uint32_t i) const
    {
        float t;
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(t) : "r"(at + i * 4u) : "memory");
        return t;
    }
};
// (past L1: other SMs wrote these entries in this very launch)
struct RowInL2 {
    const float* at;
    __device__ __forceinline__ float4 unit(int q) const { return __ldcg(reinterpret_cast<const float4*>(at) + q); }
    __device__ __forceinline__ float one(uint32_t i) const { return __ldcg(at + i); }
};
template <int K, bool kValue, typename Row>
__device__ __forceinline__ uint32_t step_of(const Row& row, double& x, float& chosen, unsigned& flags)
{
    if constexpr (K <= 4) return step16<K, false>(row, x, chosen, flags);
    else return step1<K, false, kValue>(row, x, chosen, flags);
}

// Nodes of level U go to the CTAs by fours (which then cross to a peer as one transfer): node u's CTA, its number among the nodes of its
// CTA, and back.
__device__ __forceinline__ uint32_t owner_of(uint32_t u, uint32_t mask) { return (u >> 2) & mask; }
__device__ __forceinline__ uint32_t local_of(uint32_t u, uint32_t lp) { return ((u >> (2u + lp)) << 2) | (u & 3u); }
__device__ __forceinline__ uint32_t global_of(uint32_t j, uint32_t lp, uint32_t rank) { return ((((j >> 2) << lp) + rank) << 2) | (j & 3u); }

// What a CTA stages of the levels below U: 16-byte unit q, its nodes' entries of one level after another.  (from: nullptr beyond the last, and
// for a unit beyond the level's end, which is zeroed here instead.)
struct PortionUnit { const float* from; uint32_t to; };
template <int K>
__device__ __forceinline__ PortionUnit portion_unit(const StepPlan& plan, float* portion, uint64_t min_off, uint32_t rank, uint32_t q)
{
    constexpr uint32_t lgM = kLogGroup<K>;
    PortionUnit o = PortionUnit{nullptr, 0u};
#pragma unroll 1
    for (uint32_t s = 1; s <= plan.staged; ++s) {
        const uint32_t sh = lgM * s, units = plan.own << (sh - 2u);
        if (q >= units) { q -= units; continue; }
        const uint32_t l = plan.U + s * (uint32_t)kSpan<K>, f = q * 4u, a = (global_of(f >> sh, plan.log_parts, rank) << sh) | (f & ((1u << sh) - 1u));
        const uint32_t stored = (prb_nodes_covering(plan.capacity, kLog2<K> * (plan.depth - l)) + 63u) & ~63u;
        float* const to = portion + plan.portion_at[s] + padded<K>(f);
        if (!PRB_IN_BOUNDS(plan, plan.portion_at[s] + padded<K>(f) + 4u <= plan.portion_floats)) break;
        o.to = prb_smem_addr(to);
        if (a < stored) o.from = plan.level0 + min_off + ((uint64_t)plan.off[l] << 6) + a;
        else *reinterpret_cast<float4*>(to) = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        break;
    }
    return o;
}
constexpr uint32_t kUnits = 5;                              // units of a thread whose places it looks up ahead of time

struct __align__(16) SeenLeast { double log_p; unsigned long long p_bits; };

__device__ __forceinline__ uint32_t at_rank(uint32_t smem, uint32_t rank)
{
    uint32_t to;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(smem), "r"(rank));
    return to;
}

// Rows [k0, k0 + n) of the sampled batch, as prb_copy_words; a slot among the `fresh` ones from new_lo on -- this
// launch inserts them -- is read from the insertion's batch, where that holds the field.
__device__ __forceinline__ void gather_rows(const StepPlan& plan, const PrbWordShare& g, uint32_t warps, uint32_t k0, uint32_t n,
                                            const uint32_t* s_idx, uint32_t new_lo, uint32_t fresh)
{
    const PrbWords& p = plan.out;
    const uint32_t lane = threadIdx.x & 31u, per_row = p.lane_words, at_once = 32u / per_row;
    const uint32_t stride = g.groups * at_once, r_first = g.grp * at_once + lane / per_row;
    PrbWord o = g.first;
    for (uint32_t c = g.chunk; c < p.chunks; c += warps) {
        const uint32_t w = c * 32u + (lane & (per_row - 1u));
        if (c != g.chunk) o = prb_find_word(p, w);
        if (w >= p.n_words) continue;
        unsigned char* const batch = o.batch + (uint64_t)k0 * o.batch_pitch;
        const unsigned char* in = nullptr;
        if (fresh) {
#pragma unroll
            for (int f = 0; f < PRB_NUM_FIELDS; ++f)
                if (w >= p.field[f].first) in = plan.in.field[f].batch ? plan.in.field[f].batch + ((uint64_t)(w - p.field[f].first) << p.field[f].log2) : nullptr;
        }
        constexpr int U = 4;
        for (uint32_t r0 = r_first; r0 < n; r0 += stride * U) {
            uint32_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t r = r0 + u * stride;
                if (r < n) {
                    uint32_t slot = s_idx[r];
                    if (!PRB_IN_BOUNDS(plan, slot < plan.capacity)) slot = 0u;
                    const uint32_t t = slot >= new_lo ? slot - new_lo : slot + plan.capacity - new_lo;
                    const unsigned char* at = in != nullptr && t < fresh ? in + (uint64_t)t * o.batch_pitch : o.store + (uint64_t)slot * o.store_pitch;
                    if (o.log2 == 2u) v[u] = *reinterpret_cast<const uint32_t*>(at);
                    else if (o.log2 == 1u) v[u] = *reinterpret_cast<const uint16_t*>(at);
                    else v[u] = *at;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t r = r0 + u * stride;
                if (r < n) {
                    unsigned char* at = batch + (uint64_t)r * o.batch_pitch;
                    if (o.log2 == 2u) *reinterpret_cast<uint32_t*>(at) = v[u];
                    else if (o.log2 == 1u) *reinterpret_cast<uint16_t*>(at) = (uint16_t)v[u];
                    else *at = (unsigned char)v[u];
                }
            }
        }
    }
}

// kSample: the whole iteration; otherwise the tree work (and the rows of the insertion, if they are short) alone, which only
// CTA 0 has to see the end of.  kFrames: the frame-deduplicated layout, kMin: a buffer with a
// min-tree, whose nodes go through the same steps as the sum tree's (both: tree work only).  kEach: entries of the batch, and inserted leaves, per
// thread that looks at them.
template <int K, bool kSample, bool kFrames, bool kMin, uint32_t kEach>
__global__ void __launch_bounds__(kStepThreads<kEach>, 1)
prb_step_kernel(const __grid_constant__ StepPlan plan)
{
    constexpr int M = kGroup<K>, S = kSpan<K>;
    constexpr uint32_t lg = kLog2<K>, lgM = kLogGroup<K>;
    constexpr uint32_t kThreads = kStepThreads<kEach>;
    extern __shared__ __align__(128) unsigned char s_dyn[];
    __shared__ uint32_t s_off[PRB_MAX_LEVELS];
    __shared__ uint32_t s_idx[kTreeThreads];
    __shared__ SeenLeast s_seen[kSample ? kMostSeen : 1];
    __shared__ __align__(8) unsigned long long s_bar_up, s_bar_vis, s_bar_seen;
    __shared__ unsigned s_count, s_found, s_refused;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, rank = blockIdx.x;
    const uint32_t parts = 1u << plan.log_parts, mask = parts - 1u, lp = plan.log_parts;
    float* const up = reinterpret_cast<float*>(s_dyn);
    float* const s_own = reinterpret_cast<float*>(s_dyn + plan.o_own);                         // this CTA's nodes of level U
    float* const portion = reinterpret_cast<float*>(s_dyn + plan.o_portion);
    unsigned char* const dirty = s_dyn + plan.o_dirty;
    float* const rows = reinterpret_cast<float*>(s_dyn + plan.o_rows);
    // (the min-tree's, each as far behind the sum tree's as that is long)
    float* const up_min = up + plan.up_floats;
    float* const own_min = s_own + plan.own4 * 4u;
    float* const portion_min = portion + plan.portion_floats;
    unsigned* const nodes = reinterpret_cast<unsigned*>(s_dyn + plan.o_nodes);                 // per step: keys, then the rows they have
    uint32_t* const s_place = reinterpret_cast<uint32_t*>(s_dyn + plan.o_place);               // per step and entry in hand: its group's place
    unsigned* const leaf_key = reinterpret_cast<unsigned*>(s_dyn + plan.o_leaf);
    unsigned* const leaf_last = leaf_key + plan.leaf_mask + 1u;                                // 1 + the last position that writes the leaf
    uint32_t* const l_idx = reinterpret_cast<uint32_t*>(s_dyn + plan.o_list);
    uint32_t* const l_pos = l_idx + plan.list;                                                 // (kNone: a group of the insertion)
    float* const s_val = reinterpret_cast<float*>(l_pos + plan.list);                          // value as read, then priority (negative: refused)
    uint32_t* const l_place = kEach == 1 ? l_idx : reinterpret_cast<uint32_t*>(s_val + plan.list);      // place in the leaf table, of every entry (kEach == 1: there is no list)
    const uint32_t bar_up = prb_smem_addr(&s_bar_up), bar_vis = prb_smem_addr(&s_bar_vis), bar_seen = prb_smem_addr(&s_bar_seen);
    const uint32_t N = plan.capacity, D = plan.depth;
    // strata of this CTA: its first warps', a thread each
    const uint32_t k_lo = (uint32_t)(((uint64_t)rank * plan.B) >> lp), k_hi = (uint32_t)(((uint64_t)(rank + 1u) * plan.B) >> lp);
    const uint32_t strata_warps = (((plan.B + mask) >> lp) + 31u) / 32u;         // the same in every CTA

    // ---- until the kernel before this one is complete: what depends on the arguments alone ----
    if (tid == 0) {
        const bool receives = kSample || rank == 0u;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar_up), "r"(kSample ? parts + 1u : 1u));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar_vis), "r"(parts));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_seen));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (receives) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_up), "r"((plan.n_u + 3u) / 4u * (kMin ? 32u : 16u)) : "memory");
        if (kSample) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_seen), "r"((uint32_t)sizeof(SeenLeast) * strata_warps * parts) : "memory");
        s_count = 0u; s_found = 1u; s_refused = 0u;
    }
    if (tid >= kThreads - PRB_MAX_LEVELS) s_off[tid - (kThreads - PRB_MAX_LEVELS)] = plan.off[tid - (kThreads - PRB_MAX_LEVELS)];
    {
        auto fill = [&](unsigned char* at, uint32_t bytes, uint32_t x) {      // (whole 16-byte units)
            for (uint32_t q = tid; q < bytes / 16u; q += kThreads) reinterpret_cast<uint4*>(at)[q] = make_uint4(x, x, x, x);
        };
        fill(s_dyn, plan.up_floats * (kMin ? 8u : 4u), 0u);
        fill(reinterpret_cast<unsigned char*>(s_own), plan.own4 * (kMin ? 32u : 16u), 0u);
        fill(dirty, plan.dirty_bytes, 0u);
        fill(reinterpret_cast<unsigned char*>(nodes), plan.passes * (plan.node_mask + 1u) * 4u, kNone);
        if (plan.B_upd) {
            fill(reinterpret_cast<unsigned char*>(leaf_key), (plan.leaf_mask + 1u) * 4u, kNone);
            fill(reinterpret_cast<unsigned char*>(leaf_last), (plan.leaf_mask + 1u) * 4u, 0u);
        }
    }
    constexpr uint32_t kWarps = kThreads / 32u;
    PrbWordShare share_in = {}, share_out = {};
    if (warp >= kTreeWarps && warp < kTreeWarps + kCopyThreads / 32u && plan.moves_rows) share_in = prb_word_share(plan.in, warp - kTreeWarps, kCopyThreads / 32u);
    if (kSample && warp >= strata_warps) share_out = prb_word_share(plan.out, warp - strata_warps, kWarps - strata_warps);
    if (warp < 2u) {
        // (a dry run of the arithmetic fetches its constants)
        float p = 0.0f;
        if (warp == 0u && plan.B_upd && !plan.raw && !prb_priority_pow(1.0f + (float)tid, 0.0f, 0.5f, p)) s_idx[tid] = 0u;      // (never: the square root of a small number)
        if (kSample && warp == 1u) {
            const double dry = prb_stratum_target(tid, plan.B, 1.0 + (double)tid, 0ull, plan.seed);
            if (exp2_of(-(double)plan.beta * (log2_of(2.0f + (float)dry) - 1.0)) > 1.5f) s_idx[tid] = 0u;                      // (never: 2^-x for x >= 0)
        }
    }
    // (where this thread's first units of the staged levels lie)
    PortionUnit unit[kUnits];
#pragma unroll
    for (uint32_t q = 0; q < kUnits; ++q) unit[q] = warp < kTreeWarps ? portion_unit<K>(plan, portion, 0, rank, tid + q * kTreeThreads) : PortionUnit{nullptr, 0u};
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // (every CTA's barriers can be signalled, every CTA has cleared its own memory)
    prb_dep_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const StepCtx c = StepCtx{plan, s_off};
    const uint32_t sh_u = lg * (D - plan.U);
    auto mine = [&](uint32_t leaf) { return owner_of(leaf >> sh_u, mask) == rank; };
    // the table of step p's groups: keys, then the row that holds the group
    auto keys_of = [&](uint32_t p) { return nodes + p * (plan.node_mask + 1u); };
    auto holders_of = [&](uint32_t p) { return nodes + (plan.passes + p) * (plan.node_mask + 1u); };
    const uint32_t R = plan.rows;
    auto row_at = [&](uint32_t p, uint32_t r) { return rows + (p * R + r) * kPitch<K>; };
    auto min_row_at = [&](uint32_t p, uint32_t r) { return rows + ((plan.passes + p - 1u) * R + r) * kPitch<K>; };      // (p >= 1: the leaves serve both trees)
    float* const leaves = c.level(D);
    const uint32_t n_leaves = plan.n + ((kFrames && plan.n) ? min(plan.stack, N - plan.n) : 0u);
    // group `j` of leaves that the insertion falls into, if there is such a one and it is this CTA's (else kNone); `from`: the cursor
    auto inserted_group = [&](uint32_t j, uint32_t from) {
        const bool wraps = from + n_leaves > N;
        const uint32_t a0 = from >> lgM, cnt_a = ((min(from + n_leaves, N) - 1u) >> lgM) - a0 + 1u;
        const uint32_t cnt_b = wraps && a0 ? min((from + n_leaves - N - 1u) >> lgM, a0 - 1u) + 1u : 0u;     // groups of the wrapped part not already in the first
        const uint32_t a = j < cnt_a ? a0 + j : j - cnt_a;
        return j < cnt_a + cnt_b && mine(a << lgM) ? a : kNone;
    };
    const uint32_t t256 = tid & (kTreeThreads - 1u);
    // row r for leaf i: the places of the groups above it; the first to name a group fetches it
    auto fetch = [&](uint32_t r, uint32_t i) {
        if (!PRB_IN_BOUNDS(plan, r < R && i < N)) return;
#pragma unroll 1
        for (uint32_t p = 0; p < plan.passes; ++p) {
            const uint32_t a = i >> (lgM * (p + 1u));
            unsigned* const key = keys_of(p);
            uint32_t h = prb_hash_place(a, plan.node_shift);
            unsigned old;
            while ((old = atomicCAS(key + h, kNone, a)) != kNone && old != a) h = (h + 1u) & plan.node_mask;
            s_place[p * R + r] = h;
            if (old == kNone) {
                holders_of(p)[h] = r;
                const float* const from = c.level(D - p * S) + ((uint64_t)a << lgM);
                const uint32_t to = prb_smem_addr(row_at(p, r));
                if (!PRB_IN_BOUNDS(plan, (uint64_t)a << (lgM * (p + 1u)) < N)) continue;
#pragma unroll
                for (uint32_t q = 0; q < (uint32_t)M / 4u; ++q)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + q * 16u), "l"(from + q * 4u) : "memory");
                if (kMin && p) {
                    const uint32_t to_min = prb_smem_addr(min_row_at(p, r));
#pragma unroll
                    for (uint32_t q = 0; q < (uint32_t)M / 4u; ++q)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to_min + q * 16u), "l"(from + plan.min_off + q * 4u) : "memory");
                }
            }
        }
    };
    // where the last step's node above leaf i goes: a staged level's entry (and the mark of its group), or level U's
    struct Last { float* node; unsigned char* mark; };
    auto last_of = [&](uint32_t i) {
        const uint32_t a = i >> (lgM * plan.passes), sh = lgM * plan.staged, f = (local_of(a >> sh, lp) << sh) | (a & ((1u << sh) - 1u));
        if (!PRB_IN_BOUNDS(plan, plan.staged ? plan.portion_at[plan.staged] + padded<K>(f) < plan.portion_floats && plan.dirty_at[plan.staged] + (f >> lgM) < plan.dirty_bytes
                                             : f < plan.own4 * 4u)) return Last{s_own, dirty};
        if (plan.staged == 0u) return Last{s_own + f, dirty};
        return Last{portion + plan.portion_at[plan.staged] + padded<K>(f), dirty + plan.dirty_at[plan.staged] + (f >> lgM)};
    };
    // the entry in row r, leaf i: step p's group, if it has fetched it, summed up into the next step's
    auto sum = [&](uint32_t p, uint32_t r, uint32_t i, const Last& last) {
        if (!PRB_IN_BOUNDS(plan, r < R) || holders_of(p)[s_place[p * R + r]] != r) return;
        const uint32_t a = i >> (lgM * (p + 1u)), at = a & (uint32_t)(M - 1);
        const uint32_t next = p + 1u < plan.passes ? holders_of(p + 1u)[s_place[(p + 1u) * R + r]] : 0u;
        if (!PRB_IN_BOUNDS(plan, next < R)) return;
        float e[M];
        load_group<M>(row_at(p, r), e);
        if constexpr (kMin) {
            float m[M];
            load_group<M>(p ? min_row_at(p, r) : row_at(p, r), m);
            sum_up<K, true, 0>(c, plan.min_off, D - p * S, a, m);
            if (p + 1u < plan.passes) min_row_at(p + 1u, next)[at] = m[0];
            else last.node[plan.staged ? plan.portion_floats : plan.own4 * 4u] = m[0];
        }
        sum_up<K, false, 0>(c, 0, D - p * S, a, e);
        if (p + 1u < plan.passes) {
            row_at(p + 1u, next)[at] = e[0];
        } else {
            *last.node = e[0];
            *last.mark = 1;
        }
    };
    uint32_t cursor = 0;

    if (kEach == 1 && warp >= kTreeWarps + kCopyThreads / 32u) {
        // ---- the insertion's groups: fetched and summed up like an entry's ----
        if (plan.n) cursor = (uint32_t)plan.state->cursor;
        const uint32_t j = tid - kTreeThreads - kCopyThreads, group = plan.n ? inserted_group(j, cursor) : kNone;
        if (group != kNone) fetch(kTreeThreads + j, group << lgM);
        const Last last = last_of(group != kNone ? group << lgM : 0u);
        asm volatile("cp.async.wait_all;" ::: "memory");
        copy_sync<kEach>();
        asm volatile("bar.sync 5, %0;" ::"n"(kThreads) : "memory");
        sum_sync<kEach>();
#pragma unroll 1
        for (uint32_t p = 0; p < plan.passes; ++p) {
            if (group != kNone) sum(p, kTreeThreads + j, group << lgM, last);
            sum_sync<kEach>();
        }
        cursor = __shfl_sync(0xFFFFFFFFu, cursor, 0);
        asm volatile("bar.arrive 3, %0;" ::"n"(kThreads) : "memory");
        if (!kSample) return;
    } else if (warp >= kTreeWarps) {
        // ---- entries: which are this CTA's, the groups that they fall into, the insertion's leaves; then rows ----
        int32_t ci[kEach];
        float cv[kEach], ip[kEach];
        unsigned char dn[kEach];
        const uint32_t fill = (uint32_t)plan.state->fill;
        if (plan.n || plan.stale || kFrames) cursor = (uint32_t)plan.state->cursor;
#pragma unroll
        for (uint32_t u = 0; u < kEach; ++u) {
            const uint32_t b = t256 + u * kTreeThreads;
            ci[u] = -1; cv[u] = 0.0f; ip[u] = 0.0f; dn[u] = 0;
            if (b < plan.B_upd) { ci[u] = plan.idx[b]; if (kEach > 1) cv[u] = plan.val[b]; }
            if (b < plan.n) { ip[u] = plan.prio[b]; if (kFrames) dn[u] = plan.done[b]; }
        }
        unsigned flags = 0u;
        float wmax = 0.0f;
        uint32_t take = 0;
#pragma unroll
        for (uint32_t u = 0; u < kEach; ++u) {
            if (t256 + u * kTreeThreads < plan.B_upd) {
                unsigned f = 0u;
                const bool ok = entry_ok(plan, ci[u], fill, cursor, f);
                if (rank == 0u) flags |= f;
                if (ok && mine((uint32_t)ci[u])) take |= 1u << u;
            }
        }
        uint32_t m = 0;
        if constexpr (kEach > 1) {
            const uint32_t jg = kCopyThreads - 1u - t256, group = plan.n && (jg & ~31u) <= (n_leaves >> lgM) + 2u ? inserted_group(jg, cursor) : kNone;
            // (a larger batch: this CTA's entries and groups go to a list)
            uint32_t total = 0, base = 0;
            unsigned who[kEach + 1];
#pragma unroll
            for (uint32_t u = 0; u < kEach; ++u) { who[u] = __ballot_sync(0xFFFFFFFFu, (take >> u) & 1u); total += __popc(who[u]); }
            who[kEach] = __ballot_sync(0xFFFFFFFFu, group != kNone);
            total += __popc(who[kEach]);
            if (lane == 0u && total) base = atomicAdd(&s_count, total);
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            const unsigned below = (1u << lane) - 1u;
#pragma unroll
            for (uint32_t u = 0; u < kEach; ++u) {
                const uint32_t at = base + __popc(who[u] & below);
                if (((take >> u) & 1u) && PRB_IN_BOUNDS(plan, at < plan.list)) { l_idx[at] = (uint32_t)ci[u]; l_pos[at] = t256 + u * kTreeThreads; s_val[at] = cv[u]; }
                base += __popc(who[u]);
            }
            const uint32_t at = base + __popc(who[kEach] & below);
            if (group != kNone && PRB_IN_BOUNDS(plan, at < plan.list)) { l_idx[at] = group << lgM; l_pos[at] = kNone; }
            copy_sync<kEach>();
            asm volatile("bar.arrive 7, %0;" ::"n"(kTreeThreads + kCopyThreads) : "memory");      // (the list is there: the tree warps' transform)
            m = *const_cast<volatile unsigned*>(&s_count);
        }
        // (kEach > 1: a thread holds one entry at a time; a batch that falls to few parts goes in several rounds)
#pragma unroll 1
        for (uint32_t e0 = 0;;) {
            if constexpr (kEach == 1) {
                if (take) {
                    fetch(t256, (uint32_t)ci[0]);
                    const uint32_t place = hash_find(leaf_key, plan.leaf_mask, plan.leaf_shift, (uint32_t)ci[0]);
                    atomicMax(leaf_last + place, t256 + 1u);
                    l_place[t256] = place;
                }
            } else {
                if (t256 < R && e0 + t256 < m) fetch(t256, l_idx[e0 + t256]);
                if (e0 == 0u)
                    for (uint32_t e = t256; e < m; e += kTreeThreads) {
                        if (l_pos[e] == kNone) continue;
                        const uint32_t place = hash_find(leaf_key, plan.leaf_mask, plan.leaf_shift, l_idx[e]);
                        atomicMax(leaf_last + place, l_pos[e] + 1u);
                        l_place[e] = place;
                    }
            }
            asm volatile("cp.async.wait_all;" ::: "memory");
            copy_sync<kEach>();
            // the inserted leaves of the groups in hand
            if (n_leaves) {
#pragma unroll
                for (uint32_t u = 0; u < kEach; ++u) {
                    const uint32_t t = t256 + u * kTreeThreads;
                    if (t >= n_leaves) continue;
                    const uint32_t s = cursor + t, slot = s >= N ? s - N : s, a = slot >> lgM;
                    if (!mine(slot)) continue;
                    const unsigned* const key = keys_of(0u);
                    uint32_t h = prb_hash_place(a, plan.node_shift);
                    unsigned k;
                    while ((k = key[h]) != kNone && k != a) h = (h + 1u) & plan.node_mask;
                    if (k == kNone) continue;
                    float p = 0.0f;
                    if (t < plan.n && !(kFrames && (dn[u] & kPrbEpisodeStart))) {
                        p = ip[u];
                        if (!prb_valid_priority(p)) { p = 0.0f; flags |= PEARL_ST_BAD_PRIORITY; }
                        else wmax = fmaxf(wmax, p);
                    }
                    if (!PRB_IN_BOUNDS(plan, slot < N && holders_of(0u)[h] < R)) continue;
                    row_at(0u, holders_of(0u)[h])[slot & (uint32_t)(M - 1)] = p;
                    leaves[slot] = p;
                }
            }
            asm volatile("bar.arrive 5, %0;" ::"n"(kThreads) : "memory");                  // the tree warps may go on
            if constexpr (kEach == 1) break;
            e0 += R;
            if (e0 >= m) break;
            asm volatile("bar.sync 6, %0;" ::"n"(kTreeThreads + kCopyThreads) : "memory");                    // ... and have done with these groups
            for (uint32_t h = t256; h < plan.passes * (plan.node_mask + 1u); h += kTreeThreads) nodes[h] = kNone;
            copy_sync<kEach>();
        }
        // this CTA's entries below level U are stored (and the cursor is in the hands of all its warps): every CTA that reads them, or
        // that moves the cursor, is told
        cursor = __shfl_sync(0xFFFFFFFFu, cursor, 0);
        if (warp == kTreeWarps) {
            asm volatile("bar.sync 3, %0;" ::"n"(kThreads) : "memory");
            // (Without the sample CTA 0 is told only that the others hold cursor and fill: what they have read decided their branches and
            // addresses, so it has come.  The memory model asks for a release there, too; it would wait for the leaves' stores: update and
            // insertion of 64 + 64 entries 3.60 -> 3.96 us, of 1000 + 777 5.80 -> 6.26, fanouts 2 and 16.)
            if (kSample) asm volatile("fence.acq_rel.cluster;" ::: "memory");
            if (lane < (kSample ? parts : 1u)) asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(at_rank(bar_vis, lane)) : "memory");
        } else {
            asm volatile("bar.arrive 3, %0;" ::"n"(kThreads) : "memory");
        }
        {
            const unsigned w = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(wmax));
            if (lane == 0u && w) atomicMax(&plan.state->max_prio_bits, w);
            if (flags) atomicOr(&plan.state->status, flags);
        }
        if (plan.moves_rows) {
            auto slot_from = [&](uint32_t first) {
                return [&plan, cursor, first, N](uint32_t r) {
                    const uint32_t s = cursor + first + r, slot = s >= N ? s - N : s;
                    return PRB_IN_BOUNDS(plan, slot < N && first + r < plan.n) ? slot : 0u;
                };
            };
            const uint32_t r_lo = (uint32_t)(((uint64_t)rank * plan.n) >> lp), r_hi = (uint32_t)(((uint64_t)(rank + 1u) * plan.n) >> lp);
            constexpr uint32_t kCopiers = kCopyThreads / 32u;
            if (plan.linked) prb_copy_flat(plan.in, rank * kCopiers + warp - kTreeWarps, kCopiers << lp, plan.n, slot_from(0u));
            else prb_copy_words<true>(plan.in, share_in, kCopiers, r_lo, r_hi - r_lo, slot_from(r_lo));
        }
        if (!kSample) return;
    } else {
        // ---- the tree ----
        float v0 = 0.0f;
        int32_t i0 = 0;
        if (kEach == 1 && tid < plan.B_upd) { v0 = plan.val[tid]; i0 = plan.idx[tid]; }
        const uint32_t fill = (uint32_t)plan.state->fill;
        unsigned long long calls = 0;
        if (kSample) calls = plan.state->sample_calls;
        if (plan.n || plan.stale || kFrames) cursor = (uint32_t)plan.state->cursor;
        // the staged levels of this CTA's part, and its nodes of level U (while the batch is on its way)
        float own = 0.0f;
        if (t256 < plan.own && global_of(t256, lp, rank) < plan.n_u) own = __ldcg(c.level(plan.U) + global_of(t256, lp, rank));
#pragma unroll
        for (uint32_t q = 0; q < kUnits; ++q)
            if (unit[q].from != nullptr) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(unit[q].to), "l"(unit[q].from) : "memory");
        for (uint32_t q = t256 + kUnits * kTreeThreads; q < plan.portion_units; q += kTreeThreads) {
            const PortionUnit v = portion_unit<K>(plan, portion, 0, rank, q);
            if (v.from != nullptr) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(v.to), "l"(v.from) : "memory");
        }
        float least = 0.0f;
        if constexpr (kMin) {
            if (t256 < plan.own && global_of(t256, lp, rank) < plan.n_u) least = __ldcg(c.level(plan.U) + plan.min_off + global_of(t256, lp, rank));
            for (uint32_t q = t256; q < plan.portion_units; q += kTreeThreads) {
                const PortionUnit v = portion_unit<K>(plan, portion_min, plan.min_off, rank, q);
                if (v.from != nullptr) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(v.to), "l"(v.from) : "memory");
            }
        }
        auto inserted = [&](uint32_t leaf) { return (leaf >= cursor ? leaf - cursor : leaf + N - cursor) < n_leaves; };
        unsigned flags = 0u;
        float wmax = 0.0f;
        // Priorities (negative: refused).  A small batch is transformed whole by every CTA, while the other warps find out which entries
        // are its; of a larger one each CTA transforms its own.
        auto transform = [&](float x) {
            float p = x;
            if (!(plan.raw ? prb_valid_priority(x) : prb_priority_pow(x, plan.eps, plan.alpha, p))) p = -1.0f;
            if (p < 0.0f) s_refused = 1u;
            return p;
        };
        float p0 = -1.0f;
        bool has0 = false;                       // (kEach == 1: this thread's entry is this CTA's)
        if constexpr (kEach == 1) {
            if (tid < plan.B_upd) {
                p0 = transform(v0);
                unsigned unused = 0u;
                has0 = entry_ok(plan, i0, fill, cursor, unused) && mine((uint32_t)i0);
                if (!has0) i0 = 0;
            }
        } else {
            asm volatile("bar.sync 7, %0;" ::"n"(kTreeThreads + kCopyThreads) : "memory");
            const uint32_t m = *const_cast<volatile unsigned*>(&s_count);
            for (uint32_t e = tid; e < m; e += kTreeThreads) if (l_pos[e] != kNone) s_val[e] = transform(s_val[e]);
        }
        const Last last0 = last_of((uint32_t)i0);      // (kEach == 1)
        // the leaf, if the entry is the last to write it and it is not inserted as well
        auto write_leaf = [&](uint32_t r, uint32_t i, uint32_t pos, uint32_t place, float p) {
            const uint32_t holder = holders_of(0u)[s_place[r]];
            if (p >= 0.0f) wmax = fmaxf(wmax, p);
            if (leaf_last[place] == pos + 1u && !(plan.n && inserted(i)) && PRB_IN_BOUNDS(plan, i < N && holder < R)) {
                row_at(0u, holder)[i & (uint32_t)(M - 1)] = p;
                leaves[i] = p;
            }
        };
        if (t256 < plan.own) s_own[t256] = own;
        if (kMin && t256 < plan.own) own_min[t256] = least;
        asm volatile("cp.async.wait_all;" ::: "memory");
#pragma unroll 1
        for (uint32_t e0 = 0;;) {
            asm volatile("bar.sync 5, %0;" ::"n"(kThreads) : "memory");
            const uint32_t m = kEach > 1 ? *const_cast<volatile unsigned*>(&s_count) : 0u;
            if (e0 == 0u && *const_cast<volatile unsigned*>(&s_refused)) {
                // (an entry whose priority is refused does not count as the last to write its leaf)
                for (uint32_t h = tid; h <= plan.leaf_mask; h += kTreeThreads) leaf_last[h] = 0u;
                tree_sync();
                if constexpr (kEach == 1) {
                    if (has0 && p0 >= 0.0f) atomicMax(leaf_last + l_place[tid], tid + 1u);
                    if (has0 && p0 < 0.0f) flags |= PEARL_ST_BAD_PRIORITY;
                } else {
                    for (uint32_t e = tid; e < m; e += kTreeThreads) {
                        if (l_pos[e] == kNone) continue;
                        if (s_val[e] >= 0.0f) atomicMax(leaf_last + l_place[e], l_pos[e] + 1u);
                        else flags |= PEARL_ST_BAD_PRIORITY;
                    }
                }
                tree_sync();
            }
            const bool has = kEach > 1 && tid < R && e0 + tid < m;
            uint32_t i = 0u;
            if constexpr (kEach == 1) {
                if (has0) write_leaf(tid, (uint32_t)i0, tid, l_place[tid], p0);
            } else if (has) {
                const uint32_t e = e0 + tid, pos = l_pos[e];
                i = l_idx[e];
                if (pos != kNone) write_leaf(tid, i, pos, l_place[e], s_val[e]);
            }
            sum_sync<kEach>();
            // step by step
#pragma unroll 1
            for (uint32_t p = 0; p < plan.passes; ++p) {
                if constexpr (kEach == 1) {
                    if (has0) sum(p, tid, (uint32_t)i0, last0);
                } else {
                    if (has) sum(p, tid, i, last_of(i));
                }
                sum_sync<kEach>();
            }
            if constexpr (kEach == 1) break;
            e0 += R;
            if (kEach == 1 || e0 >= m) break;
            asm volatile("bar.arrive 6, %0;" ::"n"(kTreeThreads + kCopyThreads) : "memory");
        }
        asm volatile("bar.arrive 3, %0;" ::"n"(kThreads) : "memory");
        {
            const unsigned w = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(wmax));
            if (lane == 0u && w) atomicMax(&plan.state->max_prio_bits, w);
            if (flags) atomicOr(&plan.state->status, flags);
        }
        // the staged levels: groups in which something changed
#pragma unroll 1
        for (uint32_t s = plan.staged; s > 0u; --s) {
            const uint32_t sh = lgM * (s - 1u);
            for (uint32_t g = tid; g < plan.own << sh; g += kTreeThreads) {
                const uint32_t a = (global_of(g >> sh, lp, rank) << sh) | (g & ((1u << sh) - 1u));
                if (!PRB_IN_BOUNDS(plan, plan.portion_at[s] + g * kPitch<K> + M <= plan.portion_floats && plan.dirty_at[s] + g < plan.dirty_bytes)) continue;
                float e[M];
                load_group<M>(portion + plan.portion_at[s] + g * kPitch<K>, e);
                if (!dirty[plan.dirty_at[s] + g]) continue;
                if (!PRB_IN_BOUNDS(plan, (uint64_t)a << (sh_u - sh) < N)) continue;
                if constexpr (kMin) {
                    float m[M];
                    load_group<M>(portion_min + plan.portion_at[s] + g * kPitch<K>, m);
                    sum_up<K, true, 0>(c, plan.min_off, plan.U + s * S, a, m);
                    if (s > 1u) portion_min[plan.portion_at[s - 1u] + padded<K>(g)] = m[0];
                    else own_min[g] = m[0];
                }
                sum_up<K, false, 0>(c, 0, plan.U + s * S, a, e);
                if (s > 1u) {
                    portion[plan.portion_at[s - 1u] + padded<K>(g)] = e[0];
                    dirty[plan.dirty_at[s - 1u] + (g >> lgM)] = 1;
                } else {
                    s_own[g] = e[0];
                }
            }
            tree_sync();
        }
        // The staged levels, which descents of the other CTAs read in this one's memory: one warp, behind the barrier that all who wrote them
        // have passed, releases them to every CTA's barrier.  (The transfers below do not: an asynchronous store releases
        // nothing that was written before it.)  The fence orders shared memory alone, which is all that is read before
        // bar_vis; one that waits for the stores to L2 too costs a step 0.35 us, this one less than 0.06: fanout 16, 2^20 slots, 64 + 64 entries
        // 7.69 / 7.36 / 7.35 us with it / with this one / without, 256 + 256 8.09 / 7.86 / 7.72.
        if (kSample && warp == kTreeWarps - 1u && lane < parts) {
            asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
            asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(at_rank(bar_up, lane)) : "memory");
        }
        // level U: to every CTA that goes on
        for (uint32_t t = tid; t < (kSample ? plan.own4 << lp : plan.own4); t += kTreeThreads) {
            const uint32_t peer = kSample ? t & mask : 0u, j = kSample ? t >> lp : t, u = ((j << lp) + rank) << 2;
            if (u >= plan.n_u || !PRB_IN_BOUNDS(plan, plan.up[plan.U] + u + 4u <= plan.up_floats)) continue;
            const uint4 x = reinterpret_cast<const uint4*>(s_own)[j];
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                         ::"r"(at_rank(prb_smem_addr(up + plan.up[plan.U] + u), peer)), "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w), "r"(at_rank(bar_up, peer)) : "memory");
            if constexpr (kMin) {
                const uint4 y = reinterpret_cast<const uint4*>(own_min)[j];
                asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                             ::"r"(at_rank(prb_smem_addr(up_min + plan.up[plan.U] + u), peer)), "r"(y.x), "r"(y.y), "r"(y.z), "r"(y.w), "r"(at_rank(bar_up, peer)) : "memory");
            }
        }
        if (!kSample && rank != 0u) return;
        double ku = 0.0, per_b = 0.0;
        const uint32_t k = k_lo + tid;
        if constexpr (kSample) {
            const uint32_t r0 = philox4x32_10_word0(k, 0u, (uint32_t)calls, (uint32_t)(calls >> 32), (uint32_t)plan.seed, (uint32_t)(plan.seed >> 32));
            per_b = __ddiv_rn(1.0, (double)plan.B);
            ku = __dadd_rn((double)k, __dmul_rn((double)r0, 2.3283064365386963e-10));
        }
        // the levels above U, S at a time while there are as many (what the next turn needs is looked up ahead of it); once a
        // level's nodes fit a warp the first warp goes on alone
        // (A warp one of whose threads' wait for level U was not over in time stores no sum, nor does any that sums up what other warps have summed
        // then: the barriers between them carry the answer, which as a word in shared memory cost a step 0.15 us.  In time, not late: a walk that reads
        // a peer's memory begins within one limit of polls, and the peer stays for two, see bar_seen.)
        bool sound;
        {
            uint32_t l = plan.U, h = 0, count = 0, from = 0;
            auto turn = [&]() { h = l >= (uint32_t)S ? (uint32_t)S : 1u; count = prb_nodes_covering(N, lg * (D - l + h)); from = plan.up[l]; };
            turn();
            sound = __all_sync(0xFFFFFFFFu, prb_wait_first_phase<true>(plan.state, bar_up) == kPrbInTime);
            bool alone = false;
#pragma unroll 1
            while (true) {
                if (!alone || warp == 0u)
                    for (uint32_t i = tid; i < count; i += kTreeThreads) {
                        if (h == (uint32_t)S) top_group<K, false, S>(c, up, 0, rank == 0u && sound, l, from, i);
                        else top_group<K, false, 1>(c, up, 0, rank == 0u && sound, l, from, i);
                        if constexpr (kMin) {
                            if (h == (uint32_t)S) top_group<K, true, S>(c, up_min, plan.min_off, rank == 0u && sound, l, from, i);
                            else top_group<K, true, 1>(c, up_min, plan.min_off, rank == 0u && sound, l, from, i);
                        }
                    }
                alone = alone || count <= 32u;
                l -= h;
                if (l == 0u) break;
                turn();
                if (alone) __syncwarp();
                else sound = tree_sync_all(sound);
            }
            sound = tree_sync_all(sound);
        }
        const uint64_t filled = min((uint64_t)fill + plan.n, (uint64_t)N);
        // (every CTA's warps have the cursor in hand once bar_vis is over)
        auto move_cursor = [&]() {
            if (rank != 0u || tid != 0u || plan.n == 0u) return;
            const uint32_t moved = cursor + plan.n >= N ? cursor + plan.n - N : cursor + plan.n;
            plan.state->cursor = moved;
            plan.state->fill = filled;
            if (plan.moves_rows) plan.state->row_cursor = moved;
        };
        if constexpr (!kSample) {
            if (warp == 0u && prb_wait_first_phase<true>(plan.state, bar_vis) == kPrbInTime && sound) move_cursor();
            return;
        }
        if constexpr (kSample) {
            // ---- the sample ----
            const float total32 = up[plan.up[0]];
            const double total = (double)total32;
            const bool empty = filled == 0u || !(total32 > 0.0f);
            const bool holds = k < k_hi;
            uint32_t leaf = 0;
            float p = 1.0f;
            if (warp < strata_warps) {
                unsigned wflags = 0u;
                double x = __dmul_rn(ku, total32 <= 3.402823466e+38f ? prb_quotient(total, (double)plan.B, per_b) : total);
                if (x >= total) x = __longlong_as_double(__double_as_longlong(total) - 1);
                const bool walks = holds && !empty && sound;
                uint32_t g = 0;
                if (walks) {
#pragma unroll 1
                    for (uint32_t l = 0; l < plan.U;) {
                        const uint32_t h = (plan.U - l) % (uint32_t)S ? 1u : (uint32_t)S;
                        l += h;
                        if (!PRB_IN_BOUNDS(plan, plan.up[l] + ((g + 1u) << (lg * h)) <= plan.up_floats)) g = 0u;
                        const PrbRowAt row = PrbRowAt{up + plan.up[l] + (g << (lg * h))};
                        if (h == (uint32_t)S) g = (g << lgM) + step_of<K, false>(row, x, p, wflags);
                        else g = (g << lg) + step1<K, false, false>(row, x, p, wflags);
                    }
#pragma unroll 1
                    for (uint32_t s = 1; s <= plan.staged; ++s) {
                        const uint32_t sh = lgM * (s - 1u), u = g >> sh, at_owner = (local_of(u, lp) << sh) | (g & ((1u << sh) - 1u));
                        const uint32_t local = PRB_IN_BOUNDS(plan, plan.portion_at[s] + at_owner * kPitch<K> + M <= plan.portion_floats) ? at_owner : 0u;
                        const RowOfPeer row = RowOfPeer{at_rank(prb_smem_addr(portion + plan.portion_at[s] + local * kPitch<K>), owner_of(u, mask))};
                        g = (g << lgM) + step_of<K, false>(row, x, p, wflags);
                    }
                }
                sound = prb_wait_first_phase<true>(plan.state, bar_vis) == kPrbInTime && sound;
                if (sound) move_cursor();
                if (walks && sound) {
#pragma unroll 1
                    for (uint32_t q = plan.passes; q > 0u; --q) {
                        const RowInL2 row = RowInL2{c.level(D - (q - 1u) * S) + ((uint64_t)g << lgM)};
                        if (!PRB_IN_BOUNDS(plan, (uint64_t)g << (lgM * q) < N)) { g = 0u; continue; }
                        g = (g << lgM) + step_of<K, true>(row, x, p, wflags);
                    }
                    leaf = g;
                    s_idx[tid] = leaf;
                }
                if ((tid == 0u && empty) || !sound) s_found = 0u;
                __syncwarp();
                asm volatile("bar.arrive 2, %0;" ::"n"(kThreads) : "memory");      // the copying warps may go on
                if (wflags) atomicOr(&plan.state->status, wflags);
                if (empty && sound) {
                    if (rank == 0u && tid == 0u) atomicOr(&plan.state->status, PEARL_ST_EMPTY);
                    return;
                }
                // weights: as in the sample of short rows (prb_sample_short.cu)
                const double log_p = log2_of(p);
                // (0, which no drawn leaf holds, from a thread that a wait has failed: then no CTA forms weights)
                const unsigned bits = !sound ? 0u : holds ? __float_as_uint(p) : 0x7F800000u;
                const unsigned least = __reduce_min_sync(0xFFFFFFFFu, bits);
                const double log_least = __shfl_sync(0xFFFFFFFFu, log_p, __ffs(__ballot_sync(0xFFFFFFFFu, bits == least)) - 1);
                if (lane < parts)
                    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b64 [%0], {%1, %2}, [%3];"
                                 ::"r"(at_rank(prb_smem_addr(s_seen + rank * strata_warps + warp), lane)), "l"(__double_as_longlong(log_least)), "l"((unsigned long long)least),
                                 "r"(at_rank(bar_seen, lane)) : "memory");
                if (holds && sound) plan.out_idx[k] = (int32_t)leaf;
                // (the first warp always gets here, and every walk is over when all values have come: no CTA leaves before, unless it has waited for
                // twice the limit, within which a peer that walks at all has done so)
                if (prb_wait_first_phase<true>(plan.state, bar_seen) == kPrbNever) return;
                if (rank == 0u && tid == 0u) plan.state->sample_calls = calls + 1;
                if (plan.out_w == nullptr) return;
                __syncwarp();
                unsigned best = 0xFFFFFFFFu;
                double log_best = 0.0;
                for (uint32_t j = lane; j < parts * strata_warps; j += 32u) {
                    const unsigned b = (unsigned)s_seen[j].p_bits;
                    if (b < best) { best = b; log_best = s_seen[j].log_p; }
                }
                __syncwarp();
                const unsigned smallest = __reduce_min_sync(0xFFFFFFFFu, best);
                const double log_pmin = __shfl_sync(0xFFFFFFFFu, log_best, __ffs(__ballot_sync(0xFFFFFFFFu, best == smallest)) - 1);
                if (holds && smallest != 0u) plan.out_w[k] = exp2_of(-(double)plan.beta * (log_p - log_pmin));
                return;
            }
        }
    }
    if constexpr (kSample) {
        asm volatile("bar.sync 2, %0;" ::"n"(kThreads) : "memory");
        if (s_found) gather_rows(plan, share_out, kThreads / 32u - strata_warps, k_lo, k_hi - k_lo, s_idx, cursor, plan.n);
    }
}

using StepKernel = void (*)(StepPlan);
template <bool kSample, bool kFrames, bool kMin>
StepKernel step_kernel_of(uint32_t fanout, bool many)
{
    switch (fanout) {
    case 2: return many ? prb_step_kernel<2, kSample, kFrames, kMin, kMostEach> : prb_step_kernel<2, kSample, kFrames, kMin, 1>;
    case 4: return many ? prb_step_kernel<4, kSample, kFrames, kMin, kMostEach> : prb_step_kernel<4, kSample, kFrames, kMin, 1>;
    case 8: return many ? prb_step_kernel<8, kSample, kFrames, kMin, kMostEach> : prb_step_kernel<8, kSample, kFrames, kMin, 1>;
    case 16: return many ? prb_step_kernel<16, kSample, kFrames, kMin, kMostEach> : prb_step_kernel<16, kSample, kFrames, kMin, 1>;
    default: return many ? prb_step_kernel<32, kSample, kFrames, kMin, kMostEach> : prb_step_kernel<32, kSample, kFrames, kMin, 1>;
    }
}
// form: 0 an iteration; the tree work alone: 1, with frames 2, with a min-tree 3, with both 4
constexpr uint32_t kForms = 5;
StepKernel step_kernel(uint32_t fanout, uint32_t form, bool many)
{
    switch (form) {
    case 0: return step_kernel_of<true, false, false>(fanout, many);
    case 1: return step_kernel_of<false, false, false>(fanout, many);
    case 2: return step_kernel_of<false, true, false>(fanout, many);
    case 3: return step_kernel_of<false, false, true>(fanout, many);
    default: return step_kernel_of<false, true, true>(fanout, many);
    }
}

// CTAs a cluster of this kernel may have here: 16 needs the opt-in and a group of SMs that holds it.
uint32_t most_parts(StepKernel k, uint32_t ki, uint32_t form, bool many, int dev)
{
    static uint32_t known[kPrbMaxDevices][6][kForms][2];
    uint32_t& y = known[dev][ki][form][many ? 1 : 0];
    if (y) return y;
    uint32_t most = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStepSmem) == cudaSuccess) {
        most = 8;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kStepParts);
        cfg.blockDim = dim3(many ? kStepThreads<kMostEach> : kStepThreads<1>);
        cfg.dynamicSmemBytes = kStepSmem;
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = kStepParts; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a;
        cfg.numAttrs = 1;
        int fits = 0;
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&fits, k, &cfg) == cudaSuccess && fits >= 1) most = kStepParts;
    }
    cudaGetLastError();
    y = most ? most : 1u;
    return y;
}

// Cut, staged steps and shared memory of a launch; false: a tree or batch this kernel does not take.
bool plan_step(const PrbView& v, uint32_t parts, bool many, StepPlan& p, uint32_t& smem)
{
    static_assert(kMostUpper / 4u <= kTreeThreads, "a thread each fetches a CTA's nodes of level U");
    const uint32_t S = v.fanout == 2 ? 4u : v.fanout == 4 ? 2u : 1u, lg = v.log2_fanout, lgM = lg * S, M = 1u << lgM, D = v.depth, N = (uint32_t)v.capacity;
    p.U = 0;
    for (uint32_t u = 1; u + S <= D && u < kUpperLevels; ++u)
        if ((D - u) % S == 0 && prb_nodes_covering(N, lg * (D - u)) <= (v.fanout == 32 ? kMostUpper : kMostUpper / 2u)) p.U = u;
    if (p.U == 0) return false;
    p.n_u = prb_nodes_covering(N, lg * (D - p.U));
    p.own4 = ((p.n_u + 3u) / 4u + parts - 1u) / parts;
    p.own = p.own4 * 4u;
    p.log_parts = 0;
    while ((1u << p.log_parts) < parts) ++p.log_parts;
    auto aligned = [](uint32_t x, uint32_t a) { return (x + a - 1u) / a * a; };
    uint32_t at = 0;
    for (uint32_t l = 0; l < kUpperLevels; ++l) {
        p.up[l] = at;
        if (l <= p.U) at += aligned(prb_nodes_covering(N, lg * (D - l)), M > 16u ? M : 16u);
    }
    p.up_floats = at;
    // (the staged steps stop above the leaves' own)
    const uint32_t trees = p.min_off ? 2u : 1u;
    uint32_t floats = 0, groups = 0;
    p.staged = 0;
    for (uint32_t s = 0; s <= kMostStaged; ++s) p.portion_at[s] = p.dirty_at[s] = 0;
    const uint32_t steps = (D - p.U) / S;
    for (uint32_t s = 1; s < steps && s <= kMostStaged; ++s) {
        const uint64_t here = (uint64_t)p.own << (lgM * (s - 1u));      // groups
        if ((floats + here * (M + 4u)) * trees > (many && M > 8u ? kPortionFloatsMany : kPortionFloats)) break;
        p.portion_at[s] = floats;
        p.dirty_at[s] = groups;
        floats += (uint32_t)here * (M + 4u);
        groups += (uint32_t)here;
        p.staged = s;
    }
    p.passes = steps - p.staged;
    p.portion_units = 0;
    for (uint32_t s = 1; s <= p.staged; ++s) p.portion_units += p.own << (lgM * s - 2u);
    if (p.passes > kMostPasses) return false;
    const uint32_t leaves = p.n ? p.n + p.stack : 0u;
    if (p.B_upd > kMostEntries || leaves > kMostEntries) return false;
    // (rows: a small batch's entries have one each, and after those the insertion's groups; a larger one's share kTreeThreads)
    const uint32_t groups_in = leaves ? leaves / M + 4u : 0u;
    p.list = aligned(many ? p.B_upd + groups_in : p.B_upd, 4u);
    p.rows = many ? aligned(p.list, 32u) : leaves ? kTreeThreads + aligned(groups_in, 4u) : aligned(p.B_upd, 4u);
    if (many && p.rows > kTreeThreads) p.rows = kTreeThreads;
    auto table = [](uint32_t entries, uint32_t least, uint32_t& mask, uint32_t& shift) {
        uint32_t places = least;
        shift = 32;
        while (places < 2u * entries) places *= 2u;
        for (uint32_t x = places; x > 1u; x /= 2u) --shift;
        mask = places - 1u;
    };
    table(p.B_upd, 512u, p.leaf_mask, p.leaf_shift);
    for (;; p.rows /= 2u) {
        // (fewer rows where many steps need them: what does not fit goes in rounds)
        table(many ? p.rows : p.B_upd + groups_in, 256u, p.node_mask, p.node_shift);
        uint32_t o = p.up_floats * 4u * trees;
        p.o_own = o; o = aligned(o + p.own4 * 16u * trees, 128u);
        p.portion_floats = floats;
        p.o_portion = o; o += floats * 4u * trees;
        p.dirty_bytes = aligned(groups + 1u, 16u);
        p.o_dirty = o; o += p.dirty_bytes;
        p.o_rows = o; o += (p.passes + (trees - 1u) * (p.passes - 1u)) * p.rows * (M + 4u) * 4u;
        p.o_nodes = o; o += p.passes * 2u * (p.node_mask + 1u) * 4u;
        p.o_place = o; o += p.passes * p.rows * 4u;
        p.o_leaf = o; o += p.B_upd ? 2u * (p.leaf_mask + 1u) * 4u : 0u;
        p.o_list = o; o += (many ? 4u : 1u) * p.list * 4u;
        smem = o;
        if (smem <= kStepSmem) return true;
        if (!many || p.rows <= 32u) return false;
    }
}

}  // namespace

int prb_launch_step(const PrbView& v, const PrbTreeArgs& t, const PrbSampleArgs* sample, cudaStream_t s, bool dependent)
{
    if ((sample && (v.stack || v.min_off)) || (t.n && t.prio == nullptr) || (t.B == 0 && t.n == 0)) return 0;
    PrbBatch none;
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) none.ptr[f] = nullptr;
    StepPlan p;
    p.in = prb_plan_words(v, t.rows && t.n ? *t.rows : none);
    p.out = prb_plan_words(v, sample ? sample->dst : none);
    if (p.in.n_words > kPrbMostWords || p.out.n_words > kPrbMostWords) return 0;
    const int dev = prb_current_device();
    const uint32_t form = sample ? 0u : v.min_off ? (v.stack ? 4u : 3u) : v.stack ? 2u : 1u;
    bool many = t.B > kTreeThreads || (t.n && t.n + v.stack > kTreeThreads);
    // As many CTAs as there may be -- 4 / 8 / 16, us a step: 256 + 256 entries 10.2 / 9.5 / 8.3, 1000 + 777 34 / 16.8 / 12.6; through host buffers, every CTA
    // reading the batch over the link, 40.6 / 39.1 / 37.6 -- but fewer for a small batch: the CTAs of a cluster start together, on SMs of one
    // group, and beside a learner's kernels on another stream that is what a small call waits for.  us a call, 4 / 8 / 16 CTAs, fanout 16, 2^20 slots, alone (in a
    // graph) and beside matrix products of 4096^3 in bfloat16: updates of 32 3.89 / 3.82 / 3.83 and 5.9 / 11.7 / 36; 64 + 64 4.08 / 3.95 / 3.96; steps of 32 6.76 / 6.73 /
    // 6.82 and 12 / 21 / 38; of 64 + 64 7.06 / 7.00 / 7.00 and 14 / 22 / 45.  (As two kernels 6.6 beside them for the update, 25 and 94 for the steps.)  In larger trees
    // eight CTAs have more of the tree each than they stage: fanout 4, 2^22 slots, steps of 32 10.4 / 9.9 / 9.2.
    const uint32_t entries = t.n ? t.n + v.stack : 0u, largest = sample && sample->B > entries ? sample->B : entries;
    const bool small = t.B <= 64u && largest <= 64u && v.capacity <= 1u << 20;
    const uint32_t want = t.linked ? kStepParts : !sample && t.n == 0u && t.B <= 32u ? 4u : small ? 8u : kStepParts;
    uint32_t parts = most_parts(step_kernel(v.fanout, form, many), v.log2_fanout, form, many, dev);
    if (parts > want) parts = want;
    if (parts == 1u || (sample && (sample->B > parts * kTreeThreads || sample->B > kPrbClusterStrata))) return 0;
    p.state = v.state;
    p.level0 = v.level[0];
    p.min_off = v.min_off;
    p.idx = t.idx; p.val = t.val; p.prio = t.prio; p.done = t.done;
    p.out_idx = sample ? sample->idx : nullptr;
    p.out_w = sample ? sample->w : nullptr;
    p.seed = sample ? sample->seed : 0u;
    p.capacity = (uint32_t)v.capacity;
    p.depth = v.depth;
    p.B_upd = t.B; p.n = t.n; p.B = sample ? sample->B : 1u;
    p.alpha = t.alpha; p.eps = t.eps; p.beta = sample ? sample->beta : 0.0f;
    p.raw = (uint32_t)t.raw; p.stale = t.stale; p.stack = v.stack;
    p.moves_rows = t.rows && t.n ? 1u : 0u;
    p.linked = t.linked ? 1u : 0u;
    for (uint32_t l = 0; l < PRB_MAX_LEVELS; ++l) p.off[l] = l <= v.depth ? (uint32_t)((uint64_t)(v.level[l] - v.level[0]) >> 6) : 0u;
    uint32_t smem = 0;
    if (!plan_step(v, parts, many, p, smem)) {
        // (a row for every position of the batch, and more steps than there is room for)
        if (many) return 0;
        many = true;
        parts = most_parts(step_kernel(v.fanout, form, many), v.log2_fanout, form, many, dev);
        if (parts == 1u || !plan_step(v, parts, many, p, smem)) return 0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(parts);
    cfg.blockDim = dim3(many ? kStepThreads<kMostEach> : kStepThreads<1>);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute a[2];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = parts; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
    a[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a;
    cfg.numAttrs = dependent ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, step_kernel(v.fanout, form, many), p) == cudaSuccess ? 1 : -1;
}
