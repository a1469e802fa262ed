// Tree work of a priority update and / or an insertion (PEARL Section V-A), and with short rows the insertion's
// row copy, in one launch.
//
// The update SETS leaves and re-sums their ancestors, so the result does not depend on scheduling; the last valid
// entry of the batch that names a leaf wins, and a slot that is also inserted keeps the inserted priority.
// Nothing is sorted: a batch meets in a hash table in shared memory (leaf -> last position that writes it), and
// which parents to re-sum follows from every entry by itself -- a parent reached twice is computed twice with
// the same result, an entry whose neighbour has the same parent leaves it to the neighbour.
//
// What bounds it is a chain: inputs -> transform -> leaves -> one round trip through L2 per pass over the levels
// below the staged top -> the staged levels.  So
//  * CTAs share the work by subtree: a leaf, and every node above it down to level T, belongs to the CTA that its
//    ancestor on level T falls to (round-robin), what a pass reads was written by the same CTA, and a CTA's own
//    barrier separates the passes;
//  * fanouts 2 and 4 take five and two levels per pass (a thread re-sums the 32 or 16 entries under
//    a node; with a min-tree four levels, 16 entries of either tree);
//  * an update's entries and an insertion's parents are taken from opposite ends of the CTA's threads, so that
//    their round trips overlap;
//  * levels 1 .. T (up to 20 KB) are staged in shared memory by the CTA that finishes the tree and re-summed whole
//    from there (valid because a parent always equals the sum of its children), four or two levels at a time
//    for fanouts 2 and 4; only what changed is stored.
//
// Three forms.  One CTA, or one cluster of CTAs, for up to kPrbTreeEntries update entries, one entry per thread: level T
// reaches CTA 0's staged copy through distributed shared memory, each transfer signalling a barrier there.  More entries, or a large insertion: a grid of
// CTAs, each of which picks its own entries out of the batch; the last one to finish (ticket) stages the top and
// finishes the tree.  No CTA waits for another outside its cluster.
// Launched as a programmatic dependent: until the wait nothing is read or written, the hash table is cleared and
// a dry run of the transform fetches its constants (the first use of a binary64 constant was measured at 430
// cycles, each further line of them at 84).
#include "prb_tree.cuh"
#include "prb_groups.cuh"
#include "prb_rows.cuh"

namespace {

constexpr uint32_t kTreeThreads = 1024;
constexpr uint32_t kGridThreads = 512;
constexpr uint32_t kGridList = 2048;         // entries a CTA of the grid form keeps before it works them off
constexpr int kScan = 8;                     // entries per thread and turn of its scan

struct TreePlan {
    PrbState* state;
    float* level0;
    uint64_t min_off;
    const int32_t* idx;
    const float* val;
    const float* prio;
    const unsigned char* done;
    uint32_t capacity, depth, T, top_floats;
    uint32_t B, n;                           // update entries, inserted transitions
    uint32_t raw, stale, stack;
    float alpha, eps;
    uint32_t parts, grid_form;               // CTAs of the tree work (the others copy rows)
    uint32_t many;                           // 1: passes of kPassLevels levels, 0: of one level
    uint32_t list, hash_mask, hash_shift;    // capacity of the entry list, size of the hash table less one, 32 - its log2
    uint32_t copies;                         // CTAs that copy rows
    uint32_t dependent;                      // launched as a programmatic dependent
    uint32_t linked;                         // the inputs lie in mapped host memory
    uint32_t off[PRB_MAX_LEVELS];            // level l starts off[l] * 64 entries behind level 0
    PrbWords words;
};

template <int K, bool kMin> constexpr int kPassLevels = K == 2 ? (kMin ? 4 : 5) : K == 4 ? 2 : 1;      // 32 or 16 entries under a node
template <int K> constexpr int kTopLevels = K == 2 ? 4 : K == 4 ? 2 : 1;

struct TreeCtx {
    const TreePlan& plan;
    const uint32_t* off;          // plan.off in shared memory
    float* top;                   // staged levels (CTA 0 / the last CTA), level l at (off[l] - off[1]) * 64
    float* top_min;
    uint32_t part, tid, nt;
    uint32_t bar;                 // (cluster) shared address of CTA 0's barrier, as this CTA names it: mapped to rank 0
    __device__ __forceinline__ float* level(uint32_t l) const { return plan.level0 + ((uint64_t)off[l] << 6); }
    __device__ __forceinline__ uint32_t top_at(uint32_t l) const { return (off[l] - off[1]) << 6; }
};

// Steps S .. H-1 of a block: level child-1-S and up.
template <int K, int H, int S, bool kMin>
__device__ __forceinline__ void climb(const TreeCtx& c, uint32_t child, uint32_t a, float (&e)[ipow(K, H)], float (&m)[kMin ? ipow(K, H) : 1])
{
    if constexpr (S < H) {
        constexpr int N = ipow(K, H - 1 - S);
        float* out = c.level(child - 1 - S) + (uint64_t)a * N;
        sum_groups<K, N>(e);
        store_entries<N>(out, e);
        if constexpr (kMin) {
            min_groups<K, N>(m);
            store_entries<N>(out + c.plan.min_off, m);
        }
        climb<K, H, S + 1, kMin>(c, child, a, e, m);
    }
}

// Node a of level `lt` and everything below it down to level lt+H-1, from the K^H entries of level lt+H under
// it.  (A level's end is padded with zeros to a multiple of 64 entries, so a group that reaches past it reads
// and writes zeros.)  A node of level T also goes to CTA 0's staged copy.
template <int K, int H, bool kMin>
__device__ __forceinline__ void resum(const TreeCtx& c, uint32_t lt, uint32_t a, bool staged)
{
    constexpr int M = ipow(K, H);
    const uint32_t child = lt + H;
    if (!PRB_IN_BOUNDS(c.plan, (uint64_t)a << (kLog2<K> * (c.plan.depth - lt)) < c.plan.capacity)) return;
    float e[M], m[kMin ? M : 1];
    const float* from = c.level(child) + (uint64_t)a * M;
    load_entries<M>(from, e);
    if constexpr (kMin) load_entries<M>(child == c.plan.depth ? from : from + c.plan.min_off, m);
    climb<K, H, 0, kMin>(c, child, a, e, m);
    if (staged && PRB_IN_BOUNDS(c.plan, c.top_at(lt) + a < c.plan.top_floats)) {
        const uint32_t at = c.top_at(lt) + a;
        if (c.plan.parts == 1u) {
            c.top[at] = e[0];
            if constexpr (kMin) c.top_min[at] = m[0];
        } else {
            // (a transfer that signals CTA 0's barrier: nothing else this thread has stored is waited for)
            uint32_t to;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(prb_smem_addr(c.top + at)), "r"(0u));
            asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(to), "r"(__float_as_uint(e[0])), "r"(c.bar) : "memory");
            if constexpr (kMin) {
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(prb_smem_addr(c.top_min + at)), "r"(0u));
                asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(to), "r"(__float_as_uint(m[0])), "r"(c.bar) : "memory");
            }
        }
    }
}

// Staged levels: node i of level child-H and what lies between, from the K^H staged entries under it; a group of
// nodes that comes out different is stored, staged copy and global memory.
template <int K, int H, int S>
__device__ __forceinline__ void climb_top(float* top, const TreeCtx& c, uint32_t child, uint32_t i, uint64_t min_off, float (&e)[ipow(K, H)])
{
    if constexpr (S < H) {
        constexpr int N = ipow(K, H - 1 - S);
        const uint32_t l = child - 1 - S;
        if (min_off) min_groups<K, N>(e);
        else sum_groups<K, N>(e);
        float* out = c.level(l) + min_off + (uint64_t)i * N;
        if (l == 0) {
            *out = e[0];
        } else {
            float* own = top + c.top_at(l) + i * N;
            bool same = true;
#pragma unroll
            for (int j = 0; j < N; ++j) same = same && __float_as_uint(own[j]) == __float_as_uint(e[j]);
            if (!same) { store_entries<N>(own, e); store_entries<N>(out, e); }
        }
        climb_top<K, H, S + 1>(top, c, child, i, min_off, e);
    }
}
template <int K, int H>
__device__ __forceinline__ void top_block(float* top, const TreeCtx& c, uint32_t child, uint32_t i, uint64_t min_off)
{
    constexpr int M = ipow(K, H);
    if (!PRB_IN_BOUNDS(c.plan, c.top_at(child) + (i + 1u) * M <= c.plan.top_floats)) return;
    float e[M];
    const float* from = top + c.top_at(child) + i * M;
    if constexpr (M == 2) {
        const float2 t = *reinterpret_cast<const float2*>(from);
        e[0] = t.x; e[1] = t.y;
    } else {
#pragma unroll
        for (int q = 0; q < M / 4; ++q) {
            const float4 t = reinterpret_cast<const float4*>(from)[q];
            e[4 * q] = t.x; e[4 * q + 1] = t.y; e[4 * q + 2] = t.z; e[4 * q + 3] = t.w;
        }
    }
    climb_top<K, H, 0>(top, c, child, i, min_off, e);
}

// All staged levels, from level T up to the root, by one CTA (whose threads all get here).
template <int K, bool kMin>
__device__ __forceinline__ void top_passes(const TreeCtx& c)
{
    constexpr uint32_t H = kTopLevels<K>;
    const uint32_t T = c.plan.T, D = c.plan.depth;
    for (uint32_t l = T; l > 0;) {
        // (where fewer than H levels are left a whole block is taken all the same, from levels re-summed already)
        const uint32_t h = T >= H ? H : 1u, child = max(l, h), lt = child - h;
        const uint32_t blocks = prb_nodes_covering(c.plan.capacity, kLog2<K> * (D - lt));
        for (uint32_t i = c.tid; i < blocks; i += c.nt) {
            if (h == H) top_block<K, (int)H>(c.top, c, child, i, 0);
            else top_block<K, 1>(c.top, c, child, i, 0);
            if constexpr (kMin) {
                if (h == H) top_block<K, (int)H>(c.top_min, c, child, i, c.plan.min_off);
                else top_block<K, 1>(c.top_min, c, child, i, c.plan.min_off);
            }
        }
        l = lt;
        // once a level's blocks fit a warp the first warp goes on alone
        if (blocks <= 32u) { if (c.tid >= 32u) return; __syncwarp(); }
        else __syncthreads();
    }
}

template <int K, bool kMin>
__device__ __forceinline__ void stage_top(const TreeCtx& c)
{
    const float* src = c.plan.level0 + ((uint64_t)c.plan.off[1] << 6);
    const uint32_t to = prb_smem_addr(c.top), to_min = kMin ? prb_smem_addr(c.top_min) : 0u;
    for (uint32_t q = c.tid; q < c.plan.top_floats / 4u; q += c.nt) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + q * 16u), "l"(src + q * 4u) : "memory");
        if constexpr (kMin)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to_min + q * 16u), "l"(src + c.plan.min_off + q * 4u) : "memory");
    }
}

// (kTiles: longer rows are copied as tiles; an instance of its own, so that the short rows' kernel carries none of that code)
template <int K, bool kFrames, bool kMin, bool kTiles>
__global__ void __launch_bounds__(kTreeThreads, 1)
prb_tree_kernel(const __grid_constant__ TreePlan plan)
{
    extern __shared__ __align__(16) unsigned char s_dyn[];
    __shared__ uint32_t s_off[PRB_MAX_LEVELS];
    __shared__ __align__(8) unsigned long long s_bar;        // (cluster, CTA 0) level T is complete in the staged copy
    __shared__ unsigned s_max, s_count, s_sent, s_last, s_before;
    const uint32_t tid = threadIdx.x, nt = blockDim.x;
    constexpr uint32_t lg = kLog2<K>;

    if (blockIdx.x >= plan.parts) {
        // ---- rows: the dense batch to the ring slots from row_cursor on ----
        const uint32_t c = blockIdx.x - plan.parts;
        const PrbWordShare share = prb_word_share(plan.words, tid >> 5, nt >> 5);
        prb_dep_wait();
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        const uint32_t cursor = (uint32_t)__ldcg(&plan.state->row_cursor), N = plan.capacity;
        const uint32_t r_lo = (uint32_t)(((uint64_t)c * plan.n) / plan.copies), r_hi = (uint32_t)(((uint64_t)(c + 1) * plan.n) / plan.copies);
        auto slot_from = [&](uint32_t first) {
            return [&plan, cursor, first, N](uint32_t r) {
                const uint32_t s = cursor + first + r, slot = s >= N ? s - N : s;
                return PRB_IN_BOUNDS(plan, slot < N && first + r < plan.n) ? slot : 0u;
            };
        };
        if constexpr (kTiles) prb_copy_tiles(plan.words, c, plan.copies, plan.n, slot_from(0u));
        else if (plan.linked) prb_copy_flat(plan.words, c * (nt >> 5) + (tid >> 5), plan.copies * (nt >> 5), plan.n, slot_from(0u));
        else prb_copy_words<true>(plan.words, share, nt >> 5, r_lo, r_hi - r_lo, slot_from(r_lo));
        // The ticket comes last: whoever used the cursor has had its answer (the addresses it has stored to come from it), so
        // the last CTA may move it.  (Drawn first, behind one thread's read, the rows' loads waited for the cursor, which they
        // do not need: 0.3 us an insertion.)
        __syncthreads();
        if (tid == nt - 1u && prb_ticket(&plan.state->row_ticket) == plan.copies - 1u) {
            plan.state->row_cursor = cursor + plan.n >= N ? cursor + plan.n - N : cursor + plan.n;
            plan.state->row_ticket = 0u;
        }
        return;
    }

    // ---- the tree ----
    const bool grid_form = plan.grid_form != 0u, clustered = !grid_form && plan.parts > 1u;
    TreeCtx c = TreeCtx{plan, s_off, reinterpret_cast<float*>(s_dyn), nullptr, blockIdx.x, tid, nt, 0u};
    unsigned char* at = s_dyn + plan.top_floats * sizeof(float);
    if (kMin) { c.top_min = reinterpret_cast<float*>(at); at += plan.top_floats * sizeof(float); }
    unsigned* key = reinterpret_cast<unsigned*>(at);
    unsigned* last = key + plan.hash_mask + 1u;              // 1 + the last position that writes the leaf
    uint32_t* l_idx = last + plan.hash_mask + 1u;            // this CTA's entries (several CTAs): leaf ...
    uint32_t* l_pos = l_idx + plan.list;                     // ... position in the batch
    float* l_val = reinterpret_cast<float*>(l_pos + plan.list);        // ... value, then priority
    uint32_t* l_place = reinterpret_cast<uint32_t*>(l_val + plan.list);    // ... place in the table (kNone: refused for its priority)
    float* s_prio = reinterpret_cast<float*>(l_place + plan.list);         // the inserted priorities (not in the grid form)
    auto prepare = [&]() {
        // (side by side: a warp each for what takes long, the others clear the table)
        const uint32_t w = tid >> 5;
        if (w == 0u) {
            float p = 0.0f;
            if (plan.B && !plan.raw && !prb_priority_pow(1.0f + (float)tid, 0.0f, 0.5f, p)) s_max = 1u;      // (never: the square root of a small number)
        } else if (w == 1u) {
            s_off[tid - 32u] = plan.off[tid - 32u];
        } else {
            for (uint32_t h = tid - 64u; h <= plan.hash_mask && plan.B; h += nt - 64u) { key[h] = kNone; last[h] = 0u; }
        }
        if (tid == 64u) { s_max = 0u; s_count = 0u; s_sent = 0u; s_last = 0u; s_before = 0u; }
        if (clustered) {
            if (tid == 64u && blockIdx.x == 0) {
                asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(prb_smem_addr(&s_bar)), "r"(plan.parts));
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            }
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(c.bar) : "r"(prb_smem_addr(&s_bar)), "r"(0u));
            // (relaxed: the fence above releases the barrier's initialisation, and a release here would wait for the
            // inputs' loads, slow beside a row copy: with the 512 threads below 230 -> 220 us per 8 steps of 512 rows of 56 KB)
            __syncthreads();
            asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else {
            __syncthreads();
        }
    };
    if (plan.dependent) prepare();
    prb_dep_wait();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t N = plan.capacity, D = plan.depth, T = plan.T, sh_top = min(lg * (D - T), 31u), mask = plan.parts - 1u;
    const uint32_t fill = (uint32_t)plan.state->fill;
    uint32_t cursor = 0, max_bits = 0;
    if (plan.n || plan.stale || kFrames) cursor = (uint32_t)plan.state->cursor;
    if (plan.n && plan.prio == nullptr) max_bits = plan.state->max_prio_bits;
    const uint32_t ir = nt - 1u - tid;                       // this thread's rank in the insertion's work
    int32_t i0 = -1;
    float v0 = 0.0f;
    if (!grid_form && tid < plan.B) { i0 = plan.idx[tid]; v0 = plan.val[tid]; }
    float p0 = 0.0f;
    const bool keeps_prio = !grid_form && plan.prio != nullptr;
    if (keeps_prio && tid < plan.n) p0 = plan.prio[tid];
    if (!grid_form && blockIdx.x == 0) stage_top<K, kMin>(c);

    if (!plan.dependent) prepare();                          // (nothing to hide it behind but these loads)

    // frames: the insertion also clears the leaves of the slots behind the new cursor
    const uint32_t n_leaves = plan.n + ((kFrames && plan.n) ? min(plan.stack, N - plan.n) : 0u);
    auto mine = [&](uint32_t leaf) { return ((leaf >> sh_top) & mask) == blockIdx.x; };
    auto inserted = [&](uint32_t leaf) { return (leaf >= cursor ? leaf - cursor : leaf + N - cursor) < n_leaves; };
    float* const leaves = plan.level0 + ((uint64_t)plan.off[D] << 6);
    unsigned flags = 0u;
    float wmax = 0.0f;

    // An entry's priority and, if the entry is this CTA's, its place in the table (kNone: refused).
    auto transform = [&](uint32_t i, uint32_t b, float x, float& p, bool enter) {
        p = x;
        const bool ok = plan.raw ? prb_valid_priority(x) : prb_priority_pow(x, plan.eps, plan.alpha, p);
        if (!ok) { flags |= PEARL_ST_BAD_PRIORITY; return kNone; }
        wmax = fmaxf(wmax, p);
        if (!enter) return kNone;
        const uint32_t h = hash_find(key, plan.hash_mask, plan.hash_shift, i);
        atomicMax(last + h, b + 1u);
        return h;
    };
    // New transitions without priorities take the running maximum, this update's writes included: each of several CTAs
    // then needs the whole batch's, and transforms all of it.
    const bool whole_max = plan.n != 0u && plan.prio == nullptr && plan.parts > 1u;
    // The leaf, if the entry is the last to write it (every entry has its place in the table, a barrier ago).
    auto write_leaf = [&](uint32_t i, uint32_t b, uint32_t h, float p) {
        if (h != kNone && last[h] == b + 1u && !(plan.n && inserted(i)) && PRB_IN_BOUNDS(plan, i < N)) leaves[i] = p;
    };
    // The levels between the leaves and T (a barrier after the leaves were written): `entries(one, sh)` calls one(a)
    // for the nodes a = leaf >> sh above the update's leaves; with them, the nodes above the insertion's range.
    auto passes = [&](auto entries, bool with_insertion) {
        const uint32_t h = plan.many ? (uint32_t)kPassLevels<K, kMin> : 1u;
        const uint32_t a1 = min(cursor + n_leaves, N) - 1u;                    // the inserted slots: [cursor, a1] and, wrapped, [0, b1]
        const bool wraps = cursor + n_leaves > N;
        const uint32_t b1 = wraps ? cursor + n_leaves - N - 1u : 0u;
        for (uint32_t child = D; child > T;) {
            const uint32_t lt = max(child, T + h) - h;       // (overlaps levels re-summed already where fewer than h are left)
            const uint32_t sh = min(lg * (D - lt), 31u), sh_own = lg * (lt - T);
            const bool staged = lt == T && T >= 1u && !grid_form;
            uint32_t sent = 0;
            if (clustered && lt == T) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");      // (CTA 0's staged levels are in place)
            auto one = [&](uint32_t a) {
                if (h == (uint32_t)kPassLevels<K, kMin>) resum<K, kPassLevels<K, kMin>, kMin>(c, lt, a, staged);
                else resum<K, 1, kMin>(c, lt, a, staged);
                ++sent;
            };
            entries(one, sh);
            if (with_insertion) {
                const uint32_t pa0 = cursor >> sh, cnt_a = (a1 >> sh) - pa0 + 1u;
                const uint32_t cnt_b = wraps && pa0 ? min(b1 >> sh, pa0 - 1u) + 1u : 0u;     // parents of the wrapped part not already in the first
                for (uint32_t j = ir; j < cnt_a + cnt_b; j += nt) {
                    const uint32_t a = j < cnt_a ? pa0 + j : j - cnt_a;
                    if (((a >> sh_own) & mask) == blockIdx.x) one(a);
                }
            }
            if (clustered && lt == T) {
                __syncwarp();
                sent = __reduce_add_sync(0xFFFFFFFFu, sent);
                if ((tid & 31u) == 0u && sent) atomicAdd(&s_sent, sent);
            }
            __syncthreads();
            child = lt;
        }
    };

    uint32_t m = 0, my_i = kNone, my_b = 0, my_h = kNone;      // (one entry per thread) this thread's
    float my_p = 0.0f;
    if (!grid_form) {
        bool take = false, valid = false;
        if (tid < plan.B) {
            unsigned f = 0u;
            valid = entry_ok(plan, i0, fill, cursor, f);
            if (blockIdx.x == 0) flags |= f;
            take = valid && mine((uint32_t)i0);
        }
        if (clustered && !whole_max) {
            // this CTA's entries to its first threads: the transform costs a warp the same for one entry as for 32
            const unsigned who = __ballot_sync(0xFFFFFFFFu, take);
            uint32_t base = 0;
            if (who && (tid & 31u) == 0u) base = atomicAdd(&s_count, (unsigned)__popc(who));
            base = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(who & ((1u << (tid & 31u)) - 1u));
            if (take && PRB_IN_BOUNDS(plan, base < plan.list)) { l_idx[base] = (uint32_t)i0; l_pos[base] = tid; l_val[base] = v0; }
            __syncthreads();
            valid = take = tid < s_count;
            if (take) { my_i = l_idx[tid]; my_b = l_pos[tid]; v0 = l_val[tid]; }
        } else if (valid) {
            my_i = (uint32_t)i0;
            my_b = tid;
        }
        if (valid) my_h = transform(my_i, my_b, v0, my_p, take);
        if (!take) my_i = kNone;
    } else if (plan.B) {
        // the whole batch, for the entries that are this CTA's
        if (whole_max)
            for (uint32_t b = tid; b < plan.B; b += nt) {
                unsigned unused = 0u;
                float p;
                if (entry_ok(plan, plan.idx[b], fill, cursor, unused)) transform(0u, 0u, plan.val[b], p, false);
            }
        auto work_off = [&]() {
            __syncthreads();
            const uint32_t k = s_count;
            for (uint32_t e = tid; e < k; e += nt) { float p; l_place[e] = transform(l_idx[e], l_pos[e], plan.val[l_pos[e]], p, true); l_val[e] = p; }
            __syncthreads();
            return k;
        };
        auto start_over = [&](uint32_t k) {
            for (uint32_t e = tid; e < k; e += nt) write_leaf(l_idx[e], l_pos[e], l_place[e], l_val[e]);
            __syncthreads();
            passes([&](auto one, uint32_t sh) { for (uint32_t e = tid; e < k; e += nt) one(l_idx[e] >> sh); }, false);
            for (uint32_t h = tid; h <= plan.hash_mask; h += nt) { key[h] = kNone; last[h] = 0u; }
            if (tid == 0) s_count = 0u;
            __syncthreads();
        };
        const uint32_t turn = nt * kScan, lane = tid & 31u;
        int32_t nxt[kScan];
#pragma unroll
        for (int u = 0; u < kScan; ++u) { const uint32_t b = tid + u * nt; nxt[u] = b < plan.B ? plan.idx[b] : -1; }
        for (uint32_t b0 = 0; b0 < plan.B; b0 += turn) {
            int32_t cur[kScan];
            unsigned take = 0;
#pragma unroll
            for (int u = 0; u < kScan; ++u) {
                cur[u] = nxt[u];
                const uint32_t b = b0 + turn + tid + u * nt;
                nxt[u] = b < plan.B ? plan.idx[b] : -1;      // (the next turn's, while this one's are looked at)
            }
            // (every CTA looks at the whole batch, so this loop is bound by its instructions: the index's part first;
            // range and staleness are looked at for the entries that are this CTA's, and flagged for the rows of
            // the batch that are its turn)
#pragma unroll
            for (int u = 0; u < kScan; ++u) {
                if (mine((uint32_t)cur[u])) take |= 1u << u;
                if (((b0 / nt + u) & mask) == blockIdx.x && b0 + tid + u * nt < plan.B) entry_ok(plan, cur[u], fill, cursor, flags);
            }
            uint32_t base = 0;
            if (take) {
                unsigned unused = 0u;
#pragma unroll
                for (int u = 0; u < kScan; ++u)
                    if (((take >> u) & 1u) && !(b0 + tid + u * nt < plan.B && entry_ok(plan, cur[u], fill, cursor, unused))) take &= ~(1u << u);
                base = atomicAdd(&s_count, (unsigned)__popc(take));
                const bool fits = base + (uint32_t)__popc(take) <= plan.list;
                if (!fits) s_last = 1u;                       // (0 until the tree work's end otherwise)
#pragma unroll
                for (int u = 0; u < kScan; ++u)
                    if (((take >> u) & 1u) && fits) { l_idx[base] = (uint32_t)cur[u]; l_pos[base] = b0 + tid + u * nt; ++base; }
            }
            __syncthreads();
            if (s_last) {
                // a batch that falls to few subtrees: this turn again, a row of it at a time, working the list off
                // whenever a row might not fit
                const uint32_t had = s_before;
                __syncthreads();
                if (tid == 0) { s_count = had; s_last = 0u; }
#pragma unroll
                for (int u = 0; u < kScan; ++u) {
                    __syncthreads();
                    const bool full = s_count + nt > plan.list;
                    __syncthreads();
                    if (full) start_over(work_off());
                    const unsigned who = __ballot_sync(0xFFFFFFFFu, (take >> u) & 1u);
                    uint32_t base = 0;
                    if (who && lane == 0u) base = atomicAdd(&s_count, (unsigned)__popc(who));
                    base = __shfl_sync(0xFFFFFFFFu, base, 0) + __popc(who & ((1u << lane) - 1u));
                    if (((take >> u) & 1u) && PRB_IN_BOUNDS(plan, base < plan.list)) { l_idx[base] = (uint32_t)cur[u]; l_pos[base] = b0 + tid + u * nt; }
                }
                __syncthreads();
            }
            if (tid == 0) s_before = s_count;
            __syncthreads();
        }
        m = work_off();
    }
    if (plan.n && plan.prio == nullptr) {
        // (the update's maximum: see whole_max)
        const unsigned w = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(wmax));
        if ((tid & 31u) == 0u && w) atomicMax(&s_max, w);
    }
    if (keeps_prio) {
        if (tid < plan.n) s_prio[tid] = p0;
        for (uint32_t t = tid + nt; t < plan.n; t += nt) s_prio[t] = plan.prio[t];
    }
    if (!grid_form && blockIdx.x == 0) asm volatile("cp.async.wait_all;" ::: "memory");      // (the staged levels, before any pass writes to them)
    __syncthreads();
    const float dflt = (plan.n && plan.prio == nullptr) ? prb_default_priority(max(max_bits, s_max)) : 0.0f;
    if (!grid_form) { if (my_i != kNone) write_leaf(my_i, my_b, my_h, my_p); }
    else for (uint32_t e = tid; e < m; e += nt) write_leaf(l_idx[e], l_pos[e], l_place[e], l_val[e]);
    // the inserted leaves below this CTA's nodes of level T (the slots [from, to) lie t0 behind the cursor)
    auto insert_leaves = [&](uint32_t from, uint32_t to, uint32_t t0) {
        // (one CTA: all of them at once)
        const uint32_t a_first = plan.parts == 1u ? 0u : from >> sh_top, a_last = plan.parts == 1u ? 0u : (to - 1u) >> sh_top;
        for (uint32_t a = a_first + ((blockIdx.x - a_first) & mask); a <= a_last; a += plan.parts) {
            const uint32_t lo = max(from, a << sh_top), hi = plan.parts == 1u ? to : (uint32_t)min((uint64_t)to, ((uint64_t)a + 1u) << sh_top);
            for (uint32_t slot = lo + ir; slot < hi; slot += nt) {
                const uint32_t t = slot - from + t0;
                float p = 0.0f;
                if (t < plan.n && !(kFrames && (plan.done[t] & kPrbEpisodeStart))) {
                    p = plan.prio == nullptr ? dflt : grid_form ? plan.prio[t] : s_prio[t];
                    if (!prb_valid_priority(p)) { p = 0.0f; flags |= PEARL_ST_BAD_PRIORITY; }
                    else wmax = fmaxf(wmax, p);
                }
                if (PRB_IN_BOUNDS(plan, slot < N)) leaves[slot] = p;
            }
        }
    };
    if (plan.n) {
        const uint32_t first = min(n_leaves, N - cursor);
        insert_leaves(cursor, cursor + first, 0u);
        if (first < n_leaves) insert_leaves(0u, n_leaves - first, first);
    }
    {
        const unsigned w = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(wmax));
        if ((tid & 31u) == 0u && w) atomicMax(&s_max, w);
    }
    if (flags) atomicOr(&plan.state->status, flags);
    __syncthreads();
    // CTA 0's staged levels are in place: the other CTAs, which will send their part of level T there, are told.
    // Relaxed in the ordinary build: the copies have been waited for by the threads that made them and a CTA barrier
    // has followed, so their bytes lie in CTA 0's shared memory before this arrival is issued, and what the others send
    // there is issued after they have seen it.  The memory model asks for a release, which the checked build has; it
    // would also wait for the leaves' stores (one warp releasing ahead of those stores, the others relaxed:
    // fanout 16, 2^20 slots, 1000 + 777 entries 6.49 -> 6.63 us a call).
    if (clustered) prb_cluster_arrive();
    if (tid == 0 && s_max) atomicMax(&plan.state->max_prio_bits, s_max);
    if (!grid_form) {
        passes([&](auto one, uint32_t sh) {
            // (an entry whose neighbour has the same node leaves it to the neighbour)
            const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, my_i, 1);
            if (my_i != kNone && ((tid & 31u) == 0u || before == kNone || (before >> sh) != (my_i >> sh))) one(my_i >> sh);
        }, plan.n != 0u);
    } else {
        passes([&](auto one, uint32_t sh) {
            for (uint32_t e = tid; e < m; e += nt) { const uint32_t a = l_idx[e] >> sh; if (e == 0u || (l_idx[e - 1u] >> sh) != a) one(a); }
        }, plan.n != 0u);
    }
    if (grid_form) {
        // the last CTA to finish has the whole of level T: it stages the top
        if (tid == 0) {
            __threadfence();
            s_last = prb_ticket(&plan.state->insert_ticket) == plan.parts - 1u ? 1u : 0u;
            __threadfence();
        }
        __syncthreads();
        if (!s_last) return;
        stage_top<K, kMin>(c);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (tid == 0) plan.state->insert_ticket = 0u;
    } else if (clustered) {
        // every CTA tells CTA 0's barrier how many bytes of level T it has sent there
        if (tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(c.bar), "r"(s_sent * (kMin ? 8u : 4u)) : "memory");
        if (blockIdx.x != 0) return;
        prb_wait_first_phase<false>(plan.state, prb_smem_addr(&s_bar));
        __syncthreads();
    }
    // every CTA of the tree work has read cursor and fill: they move on
    if (plan.n && tid == nt - 1u) {
        plan.state->cursor = cursor + plan.n >= N ? cursor + plan.n - N : cursor + plan.n;
        plan.state->fill = min((uint64_t)fill + plan.n, (uint64_t)N);
    }
    top_passes<K, kMin>(c);
}

using TreeKernel = void (*)(TreePlan);
template <int K, bool kTiles>
TreeKernel tree_kernel_k(bool frames, bool with_min)
{
    if (frames) return with_min ? prb_tree_kernel<K, true, true, kTiles> : prb_tree_kernel<K, true, false, kTiles>;
    return with_min ? prb_tree_kernel<K, false, true, kTiles> : prb_tree_kernel<K, false, false, kTiles>;
}
template <bool kTiles>
TreeKernel tree_kernel(const PrbView& v)
{
    const bool fr = v.stack != 0, mn = v.min_off != 0;
    switch (v.fanout) {
    case 2: return tree_kernel_k<2, kTiles>(fr, mn);
    case 4: return tree_kernel_k<4, kTiles>(fr, mn);
    case 8: return tree_kernel_k<8, kTiles>(fr, mn);
    case 16: return tree_kernel_k<16, kTiles>(fr, mn);
    default: return tree_kernel_k<32, kTiles>(fr, mn);
    }
}

constexpr uint32_t kTreeSmem = 2u * kPrbTopFloats * 4u + 2u * 2u * kGridList * 4u + 4u * kGridList * 4u + 4u * kPrbTreeEntries * 4u;      // the most a launch asks for

}  // namespace

// Which form, of the calls that prb_step.cu does not take.  One CTA while the entries' groups of a pass come to at most 2 K entries (8 KB); a cluster of 16 CTAs
// beyond -- one SM pulls and stores scattered groups so slowly that they outlast the round trip.  us a call in a graph, one CTA /
// 16: fanout 16, 48 + 48 entries 5.25 / 5.23, 96 + 96 5.5 / 5.3, 112 + 112 5.9 / 5.4; fanout 32, 48 + 48 5.6 / 5.3, 64 + 64 5.8 /
// 5.4; fanout 4, 112 + 112 6.8 / 6.5; fanout 2, 48 + 48 7.5 / 7.0, 64 + 64 7.7 / 7.0; called eagerly a single CTA is the
// cheaper launch (64 + 64: below).  us per 8 steps with
// 1 / 4 / 8 / 16 CTAs: fanout 16, 256 + 256 entries 93.3 / 83.5 / 84.0 / 80.9; fanout 2, 1000 + 777 entries 271 / 149 /
// 128 / 119; fanout 32, 512 + 512 (frames) 219 / 188 / 183 / 184; us per step at fanout 16, 64 + 64 entries 12.2 /
// 12.7 / 13.1 / 12.5, at fanout 2, 32 entries 10.9 / 11.3 / 11.7 / 11.1.  A grid beyond one entry per thread, or for an
// insertion that one CTA would take many turns to write (before it one cooperative launch with a barrier per pass and
// a launch for the insertion: 4096 + 16384 entries 56.6 -> 31.2 us a step, 4096 + 1024 41.0 -> 24.9).  Without
// priorities to read a cluster inserts up to 16384 (5000 6.4 -> 5.0 us, 16384 6.7 -> 6.1; with priorities 5000 6.5 and 6.7,
// 16384 6.8 and 11).
static bool tree_grid_form(uint32_t b, uint32_t n, bool prio) { return b > kPrbTreeEntries || n > (prio ? 4u : 16u) * kPrbTreeEntries; }
uint32_t prb_tree_ctas(const PrbView& v, uint32_t b, uint32_t n, bool prio, uint32_t most)
{
    const uint32_t group = v.fanout == 2u ? 32u : v.fanout == 4u ? 16u : v.fanout;
    const uint64_t work = (uint64_t)group * b + 4ull * n;
    const uint32_t want = tree_grid_form(b, n, prio) ? 128u : work <= 2048u ? 1u : 16u;
    return most && want > most ? most : want;
}

// Clusters beyond eight CTAs need the opt-in and a group of SMs that holds one.
static bool tree_cluster_of_16(const PrbView& v, TreeKernel k, bool tiles, int dev)
{
    static int known[kPrbMaxDevices][6][2][2][2];      // 0: not asked yet, 1: yes, 2: no
    int& y = known[dev][v.log2_fanout][v.stack ? 1 : 0][v.min_off ? 1 : 0][tiles ? 1 : 0];
    if (y == 0) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(16);
        cfg.blockDim = dim3(kTreeThreads);
        cfg.dynamicSmemBytes = kTreeSmem;
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = 16; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a;
        cfg.numAttrs = 1;
        int fits = 0;
        y = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTreeSmem) == cudaSuccess &&
            cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&fits, k, &cfg) == cudaSuccess && fits >= 1 ? 1 : 2;
        cudaGetLastError();
    }
    return y == 1;
}

int prb_launch_tree(const PrbView& v, const PrbTreeArgs& t, cudaStream_t s, bool dependent)
{
    const int dev = prb_current_device();
    if (t.B == 0 && t.n == 0) return 0;
    if (t.n && t.prio == nullptr && t.B > 2u * kPrbTreeEntries) {
        // default priorities take the update's maximum, for which every CTA would have to transform the whole batch (see
        // whole_max in the kernel): two launches from there on (4096 updates, 64 long rows: 16.3 us, 19.6 with one launch).  One launch
        // below: fanout 16, 256 + 256 entries 8.7 -> 5.3 us, 1000 + 777 10.1 -> 7.4; 2048 updates, 256 long rows 14.7 -> 13.9.
        PrbTreeArgs u = t, w = t;
        u.n = 0;
        w.B = 0;
        const int a = prb_launch_tree(v, u, s, dependent);
        const int b = a < 0 ? -1 : prb_launch_tree(v, w, s, dependent);
        return b < 0 ? -1 : a + b;
    }
    // (insertions alone that are more than a leaf a thread there: only where this file's cluster has many passes to make)
    const bool alone = t.B == 0, few = t.n + v.stack <= 256u;
    const bool deep = v.fanout == 2u || ((v.fanout == 4u || v.min_off) && v.capacity > 1u << 15);
    if (t.most_ctas == 0 && !t.linked && (!alone || few || (deep && t.n <= kTreeThreads / 2u))) {
        // up to one cluster's worth of entries in a tree that it takes (prb_step.cu).  us a call in a graph, this file's cluster / that one: fanout
        // 16, 2^20 slots, 256 entries 5.1 / 4.1, 256 + 256 5.6 / 4.4, 64 + 64 5.4 / 4.1, 256 insertions 4.1 / 3.5; fanout 2, 1000 + 777 8.9 / 6.2;
        // fanout 32, 2^22 slots, 1024 + 1024 7.7 / 6.4 -- and 1024 insertions alone 5.4 / 5.9: their rows are better copied by CTAs of their own.  400
        // insertions alone: fanout 2, 2^15 slots 5.3 / 4.5; 4, 2^20 slots 5.0 / 4.3; 8, 2^20 slots 4.5 / 5.2; 16, 3000 slots 3.3 / 3.8; 32, 2^15 slots 3.65 / 4.06; with a
        // min-tree 512 at fanout 8, 2^20 slots 5.6 / 5.1, at 32, 2^15 slots 4.65 / 4.83; 4, 3000 slots 3.63 / 3.84.  Fanouts 4 and 8, 2^18 slots, 64 + 64 entries:
        // 5.6 / 3.9 and 5.0 / 4.1.
        const int k = prb_launch_step(v, t, nullptr, s, dependent);
        if (k != 0) return k;
    }
    TreePlan p;
    p.state = v.state;
    p.level0 = v.level[0];
    p.min_off = v.min_off;
    p.idx = t.idx; p.val = t.val; p.prio = t.prio; p.done = t.done;
    p.capacity = (uint32_t)v.capacity;
    p.depth = v.depth;
    p.B = t.B; p.n = t.n;
    p.raw = (uint32_t)t.raw; p.stale = t.stale; p.stack = v.stack;
    p.alpha = t.alpha; p.eps = t.eps;
    for (uint32_t l = 0; l < PRB_MAX_LEVELS; ++l) p.off[l] = l <= v.depth ? (uint32_t)((uint64_t)(v.level[l] - v.level[0]) >> 6) : 0u;
    // T: the deepest level that fits the staging area and leaves a whole pass below it
    const uint32_t h = v.fanout == 2 ? (v.min_off ? 4u : 5u) : v.fanout == 4 ? 2u : 1u;
    p.many = v.depth > h ? 1u : 0u;
    const uint32_t below = p.many ? h : 1u;
    p.T = 0;
    p.top_floats = 0;
    for (uint32_t l = 1; l + below <= v.depth; ++l) {
        const uint64_t end = ((uint64_t)(p.off[l] - p.off[1]) << 6) + (v.level_alloc[l] + 63u) / 64u * 64u;
        if (end > kPrbTopFloats) break;
        p.T = l;
        p.top_floats = (uint32_t)end;
    }
    PrbBatch none;
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) none.ptr[f] = nullptr;
    p.words = prb_plan_words(v, t.rows ? *t.rows : none);
    const bool tiles = p.words.n_words > kPrbMostWords && !t.linked;
    const TreeKernel k = tiles ? tree_kernel<true>(v) : tree_kernel<false>(v);
    p.grid_form = tree_grid_form(t.B, t.n, t.prio != nullptr) ? 1u : 0u;
    uint32_t parts = p.T ? prb_tree_ctas(v, t.B, t.n, t.prio != nullptr, t.most_ctas) : 1u;      // (no staged level: nothing to split by)
    // (an insertion of longer rows alone: its copying CTAs, which take longer than the tree work, would come in clusters, too,
    // and leave SMs idle that no whole cluster fits on: 1024 rows of 14 KB 9.3 us with a cluster of 16, 6.8 with one CTA)
    if (tiles && t.B == 0u && !p.grid_form) parts = 1u;
    p.parts = parts;
    p.list = p.grid_form ? kGridList : t.B;
    // (at least 512 places, whatever the entries: probes are a chain of shared atomics; 32 entries in 64 places took 4.7 to
    // 5.5 us a call, by the batch's luck)
    uint32_t slots = 512;
    p.hash_shift = 23;
    while (slots < 2u * p.list) { slots *= 2u; --p.hash_shift; }
    p.hash_mask = t.B ? slots - 1u : 0u;
    if (t.B == 0) p.list = 0;
    // (grid: what a large batch costs is that every CTA looks at all of it.  fanout 16, with 1024 insertions, 512 / 1024 threads:
    // 4096 entries 9.7 / 10.4 us a call, 8192 11.4 / 10.4, 16384 15.1 / 12.3, 49000 28.7 / 19.8)
    uint32_t threads = t.B >= 8u * kPrbTreeEntries ? kTreeThreads : kGridThreads;
    if (!p.grid_form) {
        threads = (t.B + 31u) / 32u * 32u + (t.n < 512u ? (t.n + 31u) / 32u * 32u : 512u);
        threads = threads < 256u ? 256u : threads > kTreeThreads ? kTreeThreads : threads;
        // Beside a row copy no more than an entry each asks for: a copying CTA holds 20480 of an SM's 65536 registers, and
        // 512 of these threads hold 32768, so that the cluster fits on SMs that copy too.  With 1024 it needed whole SMs, eight
        // of them in one group (512 + 512 entries alone with their rows: 10.1 us, 9.85 this way).
        if (t.most_ctas == kPrbTreeBesideRows && threads > 512u) threads = t.B <= 512u ? 512u : (t.B + 31u) / 32u * 32u;
    }
    p.copies = 0;
    p.dependent = dependent ? 1u : 0u;
    p.linked = t.linked ? 1u : 0u;
    if (t.rows && t.n) {
        // a few rows' words per warp, or a tile per CTA, on the SMs the tree work leaves
        uint64_t ctas = 0;
        if (tiles) {
            for (int f = 0; f < PRB_NUM_FIELDS; ++f) ctas += ((uint64_t)t.n * p.words.field[f].units() + kPrbTile - 1) / kPrbTile;
        } else {
            const uint64_t items = (uint64_t)t.n * p.words.chunks * p.words.lane_words / 32u, per_cta = threads / 32u * 4u;
            ctas = (items + per_cta - 1) / per_cta;
            if (ctas > t.n) ctas = t.n;
        }
        const uint64_t room = (uint64_t)prb_sm_count() * (threads <= 512u ? 2u : 1u) - parts;
        if (ctas > room) ctas = room;
        p.copies = ctas ? (uint32_t)ctas : 1u;
    }
    if (!p.grid_form && parts > 8u && !tree_cluster_of_16(v, k, tiles, dev)) p.parts = parts = 8u;
    const uint32_t cluster = p.grid_form ? 1u : parts;
    p.copies = p.copies ? (p.copies + cluster - 1u) / cluster * cluster : 0u;      // (whole clusters)
    static bool ready[kPrbMaxDevices][6][2][2][2];
    bool& rd = ready[dev][v.log2_fanout][v.stack ? 1 : 0][v.min_off ? 1 : 0][tiles ? 1 : 0];
    if (!rd) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTreeSmem) != cudaSuccess) return -1;
        rd = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(parts + p.copies);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = p.top_floats * 4u * (v.min_off ? 2u : 1u) + (t.B ? 2u * (p.hash_mask + 1u) * 4u : 8u) + 4u * p.list * 4u +
                           (p.grid_form || t.prio == nullptr ? 0u : (t.n + 3u) / 4u * 16u);
    cfg.stream = s;
    cudaLaunchAttribute a[2];
    uint32_t na = 0;
    if (cluster > 1u) {
        a[na].id = cudaLaunchAttributeClusterDimension;
        a[na].val.clusterDim.x = cluster; a[na].val.clusterDim.y = 1; a[na].val.clusterDim.z = 1;
        ++na;
    }
    if (dependent) {
        a[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        a[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    cfg.attrs = a;
    cfg.numAttrs = na;
    return cudaLaunchKernelEx(&cfg, k, p) == cudaSuccess ? 1 : -1;
}
