// Batched insertion: ring write of n transitions into the Data Storage and the matching
// leaf writes + ancestor re-sum in the sum tree (PEARL Section V-A: insertion is realised as
// priority retrieval followed by priority update; Listing 2: experiences are added to the
// Data Storage and insertion requests go to the Replay Manager).
//
// Short rows: one launch of the tree kernel (prb_tree.cu), whose spare CTAs copy them.
// Long rows (at least 8 KB of 16-byte granules, Atari-shaped): the kernel below, one CTA per SM; warp 0 of
// every CTA drives bulk asynchronous copies global -> shared -> global through a ~200 KB
// ring (row chunks of <= 8 KB, one lane per stage), issuing its loads before the cursor has
// even arrived; the other warps copy the short fields.  CTA 0 does the tree and moves no rows;
// with a priority update in the same call the tree work is the tree kernel's, beside this one, and every
// CTA here copies.
// Tree work here: write the n leaves, then re-sum the dirty parents level by level (a contiguous
// slot range dirties a contiguous parent range on every level, so no sorting is needed).
// The CTA that is last to have read the cursor advances it (and the fill count) while the copies
// are still running.  No CTA waits on another.
#include "prb_tree.cuh"

namespace {

constexpr int kWorkers = 256;                // threads that copy short rows / do the tree work
constexpr int kThreadsRows = 32 + kWorkers + 32; // long-row kernel: ring warp, workers, publishing warp
constexpr uint32_t kChunk = 512;             // upper bound on granules per chunk of a long row (8 KB)
constexpr uint32_t kTile = kWorkers * 8;     // granules per tile of short rows
constexpr uint32_t kRowMode = 512;           // rows of at least this many 16-byte granules are split into chunks
constexpr uint32_t kRingBytes = 198 * 1024;  // bulk-copy ring (dynamic shared memory), <= 32 stages
constexpr uint32_t kRingBarBytes = 1024;     // room for the ring's mbarriers in front of its buffers
// Bytes of long rows from which the tree work goes to the side stream.  Rows of 56 KB, us a call / a step with the fork and
// without: 32 6.4 / 14.5 and 6.4 / 14.3, 128 6.5 / 15.4 and 6.6 / 15.2, 256 7.1 / 17.1 and 7.2 / 17.2, 512 9.3 / 25.6 and 12.4 / 29.6:
// the same up to 256, and called eagerly the fork costs two events (4 rows: 18.6 -> 16.9 us a step without).
constexpr uint64_t kForkFrom = 4ull << 20;

struct InsertPlan {
    // short-row tiles, numbered field by field: tiles of field f are [first_tile[f], first_tile[f+1])
    uint32_t first_tile[PRB_NUM_FIELDS + 1];
    // long-row tasks (one chunk of one row), numbered field by field
    uint32_t first_task[PRB_NUM_FIELDS + 1];
    uint32_t chunks[PRB_NUM_FIELDS];          // chunks per row of a long-row field, else 0
    uint32_t chunk[PRB_NUM_FIELDS];           // granules per chunk
    uint32_t ring_stages, ring_stage_bytes;
    // CTAs of a tree kernel that runs beside this one and does the insertion's tree work (0: this
    // kernel does it); this kernel then keeps the row cursor, with a ticket of its own
    uint32_t tree_ctas;
};

// Short rows: tile `tile` of the dense batch of field f, which may span many rows.
template <typename T>
__device__ __forceinline__ void copy_flat_tile(const PrbView& v, int f, const PrbBatch& src, uint32_t n, uint64_t cursor,
                                               uint32_t tile, uint32_t rank, uint32_t nthreads)
{
    const uint32_t W = v.field_bytes[f] / sizeof(T), Wp = v.field_pitch[f] / sizeof(T);     // granules per row, per slot of the store
    const uint64_t N = v.capacity;
    const uint64_t total = (uint64_t)n * W;
    const uint64_t e0 = (uint64_t)tile * kTile;
    const uint32_t e1 = (uint32_t)min(total, e0 + kTile);
    prb_copy_mapped<T>(reinterpret_cast<T*>(v.store[f]), reinterpret_cast<const T*>(src.ptr[f]), (uint32_t)e0, e1,
                       [=](uint32_t e) { return (uint64_t)e; },
                       [=](uint32_t e) {
                           const uint32_t r = e / W;
                           uint64_t slot = cursor + r;
                           if (slot >= N) slot -= N;
                           if (!PRB_IN_BOUNDS(v, slot < N && r < n)) slot = 0;
                           return slot * Wp + (e - r * W);
                       },
                       rank, nthreads);
}

__device__ __forceinline__ void copy_tile(const PrbView& v, const InsertPlan& plan, const PrbBatch& src, uint32_t n,
                                          uint64_t cursor, uint32_t tile, uint32_t rank, uint32_t nthreads)
{
    int f = 0;
    while (tile >= plan.first_tile[f + 1]) ++f;
    const uint32_t local = tile - plan.first_tile[f];
    switch (v.field_vec[f]) {
    case 16: copy_flat_tile<uint4>(v, f, src, n, cursor, local, rank, nthreads); break;
    case 8: copy_flat_tile<uint2>(v, f, src, n, cursor, local, rank, nthreads); break;
    case 4: copy_flat_tile<uint32_t>(v, f, src, n, cursor, local, rank, nthreads); break;
    case 2: copy_flat_tile<uint16_t>(v, f, src, n, cursor, local, rank, nthreads); break;
    default: copy_flat_tile<uint8_t>(v, f, src, n, cursor, local, rank, nthreads); break;
    }
}

// Long rows present.  Warp 0: lane s owns ring stage s and moves row chunks t_lo+s, t_lo+s+S, ...
// of this CTA's range; the first loads go out before the cursor has arrived (a source address does
// not depend on it).  Threads 32..32+kWorkers-1: the tree work (CTA 0, unless a tree kernel beside
// this one does it) and the short-field tiles (dealt round-robin, CTA 1 first).  Thread
// 32+kWorkers: cursor and ticket.
template <bool kFrames, bool kMin>
__global__ void __launch_bounds__(kThreadsRows, 1)
prb_insert_rows_kernel(const __grid_constant__ PrbView v, uint32_t n, const __grid_constant__ PrbBatch src,
                       const float* __restrict__ prio, const __grid_constant__ InsertPlan plan)
{
    extern __shared__ __align__(128) unsigned char s_ring[];
    __shared__ unsigned long long s_cursor, s_fill;     // read once per CTA, before anything is published
    __shared__ unsigned int s_maxp;                     // running maximum of priorities at kernel start
    const uint32_t tid = threadIdx.x;
    const uint32_t n_tasks = plan.first_task[PRB_NUM_FIELDS];
    // A CTA that does the tree work moves no rows: the answers to its tree reads would queue behind
    // the data of its own bulk loads.
    const uint32_t first_copy_cta = (plan.tree_ctas == 0 && gridDim.x > 1) ? 1u : 0u;
    const uint32_t copy_ctas = gridDim.x - first_copy_cta;
    const bool copies = blockIdx.x >= first_copy_cta;
    const uint32_t cc = blockIdx.x - first_copy_cta;
    const uint32_t t_lo = copies ? (uint32_t)(((uint64_t)cc * n_tasks) / copy_ctas) : 0u;
    const uint32_t t_hi = copies ? (uint32_t)(((uint64_t)(cc + 1) * n_tasks) / copy_ctas) : 0u;
    const bool ring_lane = copies && tid < plan.ring_stages;
    constexpr uint32_t kPublisher = 32 + kWorkers;

    // one row chunk: field, row in the batch, first granule, bytes
    auto locate = [&](uint32_t t, int& f, uint32_t& row, uint32_t& W, uint32_t& e0, uint32_t& bytes) {
        f = 0;
        while (t >= plan.first_task[f + 1]) ++f;
        const uint32_t local = t - plan.first_task[f];
        row = local / plan.chunks[f];
        W = v.field_bytes[f] / 16u;
        e0 = (local - row * plan.chunks[f]) * plan.chunk[f];
        bytes = min(W - e0, plan.chunk[f]) * 16u;
    };

    PrbBulkLane ring;
    int f = 0; uint32_t row = 0, W = 0, e0 = 0, bytes = 0;
    uint32_t t = t_lo + tid;
    // (beside a tree kernel this kernel keeps the row cursor only: see PrbState)
    if (tid == kPublisher) { s_cursor = plan.tree_ctas ? v.state->row_cursor : v.state->cursor; s_fill = v.state->fill; s_maxp = v.state->max_prio_bits; }
    if (ring_lane) {
        ring.init(s_ring + 8u * tid, s_ring + kRingBarBytes + tid * plan.ring_stage_bytes);
        if (t < t_hi) {
            locate(t, f, row, W, e0, bytes);
            ring.load(src.ptr[f] + ((uint64_t)row * W + e0) * 16u, bytes);
        }
    }
    __syncthreads();
    const uint64_t cursor = s_cursor;

    if (tid == kPublisher) {
        prb_publish_if_last(v, n, cursor, s_fill, gridDim.x, plan.tree_ctas ? kPrbPublishRows : kPrbPublishAll);
    } else if (ring_lane) {
        while (t < t_hi) {
            uint64_t slot = cursor + row;
            if (slot >= v.capacity) slot -= v.capacity;
            if (!PRB_IN_BOUNDS(v, slot < v.capacity && row < n && e0 < W && bytes <= plan.ring_stage_bytes)) slot = 0;
            ring.store(v.store[f] + (slot * W + e0) * 16u, bytes);
            t += plan.ring_stages;
            if (t < t_hi) {
                locate(t, f, row, W, e0, bytes);
                ring.load(src.ptr[f] + ((uint64_t)row * W + e0) * 16u, bytes);
            }
        }
        ring.finish();
        if (ring.failed) atomicOr(&v.state->status, PEARL_ST_INTERNAL);
    } else if (tid >= 32 && tid < kPublisher) {
        PrbTeam team;
        team.rank = tid - 32u; team.size = kWorkers; team.whole_cta = false;
        if (kMin) team.min_off = v.min_off;
        if (blockIdx.x == 0 && plan.tree_ctas == 0)
            prb_insert_tree_team(v, team, n, prio, cursor, s_maxp, src.ptr[F_DONE],
                                 kFrames ? v.stack : 0u);
        const uint32_t n_tiles = plan.first_tile[PRB_NUM_FIELDS];
        for (uint32_t tile = (blockIdx.x + gridDim.x - 1) % gridDim.x; tile < n_tiles; tile += gridDim.x)
            copy_tile(v, plan, src, n, cursor, tile, team.rank, team.size);
    }
    // Launched as a programmatic dependent of the tree kernel: this kernel is complete only when that one is.
    prb_dep_wait();
}

}  // namespace

int prb_launch_insert(const PrbView& v, uint32_t n, const PrbBatch& src, const float* d_prio, cudaStream_t s,
                      uint32_t upd_B, const int32_t* upd_idx, const float* upd_val, int upd_raw, float alpha, float eps,
                      const PrbFork* fork, bool* beside_out, bool rows_only, bool linked)
{
    if (beside_out) *beside_out = false;
    if (rows_only && upd_B) return -1;
    const int sm_count = prb_sm_count();
    const int dev = prb_current_device();
    PrbTreeArgs tree;
    tree.B = upd_B; tree.idx = upd_idx; tree.val = upd_val; tree.raw = upd_raw; tree.alpha = alpha; tree.eps = eps;
    tree.n = n; tree.prio = d_prio; tree.done = src.ptr[F_DONE];

    InsertPlan plan;
    uint32_t tiles = 0, tasks = 0, stage = 0;
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) {
        plan.first_tile[f] = tiles;
        plan.first_task[f] = tasks;
        plan.chunks[f] = 0;
        plan.chunk[f] = 0;
        if (v.field_bytes[f] == 0 || src.ptr[f] == nullptr) continue;
        const uint32_t W = v.field_bytes[f] / v.field_vec[f];
        if (v.field_vec[f] == 16 && W >= kRowMode) {
            plan.chunks[f] = (W + kChunk - 1) / kChunk;
            plan.chunk[f] = (W + plan.chunks[f] - 1) / plan.chunks[f];
            tasks += n * plan.chunks[f];
            if (plan.chunk[f] * 16u > stage) stage = plan.chunk[f] * 16u;
        } else {
            const uint64_t total = (uint64_t)n * W;
            tiles += (uint32_t)((total + kTile - 1) / kTile);
        }
    }
    if (rows_only && tasks == 0) return -1;
    int ahead = 0;      // launches ahead of the insertion's
    // a very large update goes first, in a launch of its own: also one that is two launches anyway (no priorities, see
    // prb_launch_tree) or that eight CTAs beside a copy of long rows would work on (16384 entries, 32 rows: 26 us a call, 14 this way)
    if (upd_B && (prb_update_is_wide(v, upd_B, d_prio != nullptr) || (tasks && upd_B > 4u * kPrbTreeEntries))) {
        ahead = prb_launch_update_wide(v, upd_B, upd_idx, upd_val, upd_raw, alpha, eps, s, 0u);
        if (ahead < 0) return -1;
        if (ahead) tree.B = upd_B = 0;
    }
    if (tasks == 0) {
        // short rows: one launch does the update, the insertion's tree work and the row copy
        tree.rows = &src;
        tree.linked = linked;
        // (every CTA reads the indices over the link; a larger update's have been copied to the device: with 4 CTAs all the
        // same, a host step of 4000 updates and 64 insertions took 70 us and one of 5000 updates 78, 61 and 65 without the limit)
        if (linked && upd_B <= kPrbTreeEntries) tree.most_ctas = 4u;
        const int k = prb_launch_tree(v, tree, s, true);
        return k < 0 ? -1 : ahead + k;
    }
    plan.first_tile[PRB_NUM_FIELDS] = tiles;
    plan.first_task[PRB_NUM_FIELDS] = tasks;
    plan.tree_ctas = 0;
    stage = (stage + 127u) / 128u * 128u;
    plan.ring_stage_bytes = stage;
    plan.ring_stages = kRingBytes / stage;
    if (plan.ring_stages > 32) plan.ring_stages = 32;
    int launches = 1;
    const bool beside = upd_B != 0;
    bool forked = false;
    // Without a tree kernel CTA 0 does the tree work and no copies; with one, its CTAs get SMs of
    // their own: a copy CTA takes an SM's whole shared memory and would wait for them to leave.
    const uint32_t want = tasks + ((beside || rows_only) ? 0u : 1u);
    uint32_t room = (uint32_t)sm_count;
    if (rows_only) {
        plan.tree_ctas = 1;       // (CTA 0 copies like the others and the row cursor is published by itself)
    } else if (beside) {
        // The update and the insertion's tree work are one kernel, the row copy another beside it; neither waits for
        // the other (each advances a cursor of its own).  (In one kernel the tree's chain of dependent reads, slowed
        // by the copy's traffic, was measured to outlast the copy by far.)
        // Few rows: both on the caller's stream, the copy a programmatic dependent that does not wait: it starts as
        // soon as the tree kernel's CTAs have (they have waited for what came before) and waits for the tree only
        // before it ends, so that what follows has both behind it.  No fork, no join: 4 rows of 56 KB, 18.6 ->
        // 16.9 us a step.  Many rows: the tree kernel on the side stream, so that the copy, the longer of the two,
        // does not start behind the tree kernel's start (512 rows of 56 KB: 33.5 us a step the first way).
        forked = fork != nullptr && (uint64_t)tasks * stage > kForkFrom;
        tree.most_ctas = kPrbTreeBesideRows;
        plan.tree_ctas = prb_tree_ctas(v, upd_B, n, d_prio != nullptr, tree.most_ctas);
        if (room > 2u * kPrbTreeBesideRows) room -= kPrbTreeBesideRows;
        if (forked && (cudaEventRecord(fork->fork, s) != cudaSuccess || cudaStreamWaitEvent(fork->side, fork->fork, 0) != cudaSuccess)) return -1;
        const int k = prb_launch_tree(v, tree, forked ? fork->side : s, !forked);
        if (k < 1 || (forked && cudaEventRecord(fork->join, fork->side) != cudaSuccess)) return -1;
        launches = 1 + k;
        if (beside_out) *beside_out = true;
    }
    const uint32_t rows_grid = want < room ? want : room;
    const uint32_t smem = kRingBarBytes + plan.ring_stages * plan.ring_stage_bytes;
    static bool big_rows[kPrbMaxDevices];
    if (!big_rows[dev]) {
        bool ok = true;
#define PRB_ALLOW_SMEM(FF, MM) \
    ok = ok && cudaFuncSetAttribute(prb_insert_rows_kernel<FF, MM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kRingBarBytes + kRingBytes)) == cudaSuccess
        PRB_ALLOW_SMEM(false, false); PRB_ALLOW_SMEM(true, false); PRB_ALLOW_SMEM(false, true); PRB_ALLOW_SMEM(true, true);
#undef PRB_ALLOW_SMEM
        if (!ok) return -1;
        big_rows[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(rows_grid);
    cfg.blockDim = dim3(kThreadsRows);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = beside && !forked ? 1 : 0;
    cudaError_t e = cudaSuccess;
#define PRB_LAUNCH_ROWS_AS(FF, MM) e = cudaLaunchKernelEx(&cfg, prb_insert_rows_kernel<FF, MM>, v, n, src, d_prio, plan)
    PRB_WITH_TREE_OPTIONS(v, PRB_LAUNCH_ROWS_AS);
#undef PRB_LAUNCH_ROWS_AS
    if (e != cudaSuccess || (forked && cudaStreamWaitEvent(s, fork->join, 0) != cudaSuccess)) return -1;
    return ahead + launches;
}
