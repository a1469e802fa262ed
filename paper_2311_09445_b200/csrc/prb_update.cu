// Batched changes of priorities (PEARL Section V-A's own interface: index + change) and priority retrieval.  Values
// and TD errors are set by the tree kernel (prb_tree.cu); changes add up in batch order, so their batch is sorted
// (see prb_delta_team in prb_tree.cuh for the steps).  One CTA, or eight CTAs of one thread-block cluster that
// share the deep levels.
#include "prb_tree.cuh"

namespace {

// kFrames: the instance for the frame-deduplicated layout (stale history-less updates)
// kMin: the instance that maintains the min-tree beside the sum tree
template <bool kFrames, bool kMin>
__global__ void __launch_bounds__(1024)
prb_delta_kernel(const __grid_constant__ PrbView v, uint32_t B, uint32_t n2, const int32_t* __restrict__ idx,
                 const float* __restrict__ val)
{
    extern __shared__ __align__(16) unsigned char smem[];
    // (a programmatic dependent behind this kernel may be made resident now; it waits for this kernel's
    // completion before it reads anything)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    PrbTeam team;
    team.rank = threadIdx.x;
    team.size = blockDim.x;
    team.whole_cta = true;
    team.part = blockIdx.x;          // CTAs of one cluster share the work (one CTA: the whole of it)
    team.parts = gridDim.x;
    if (kMin) team.min_off = v.min_off;
    PrbTop top;
    if (v.top_levels) top.mem = reinterpret_cast<float*>(smem + prb_update_smem_bytes(n2));
    if (kMin && v.top_levels) top.mem_min = top.mem + v.top_floats;
    if (team.part == 0) prb_top_begin(v, top, team.rank, team.size);
    const unsigned long long fill = v.state->fill;
    prb_delta_team(v, team, B, n2, idx, val, fill, smem, kFrames ? v.state->cursor : 0ull, top, kFrames ? v.stack : 0u);
}

// Priority retrieval: one thread per entry.
__global__ void prb_get_priorities_kernel(const __grid_constant__ PrbView v, uint32_t B, const int32_t* __restrict__ idx,
                                          float* __restrict__ out)
{
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int32_t i = idx[b];
    if (i < 0 || (unsigned long long)i >= v.state->fill) { out[b] = 0.0f; atomicOr(&v.state->status, PEARL_ST_BAD_INDEX); return; }
    out[b] = PRB_IN_BOUNDS(v, (uint32_t)i < v.level_alloc[v.depth]) ? __ldcg(v.level[v.depth] + i) : 0.0f;
}

}  // namespace

int prb_launch_get_priorities(const PrbView& v, uint32_t B, const int32_t* d_idx, float* d_out, cudaStream_t s)
{
    prb_get_priorities_kernel<<<(B + 255) / 256, 256, 0, s>>>(v, B, d_idx, d_out);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

uint32_t prb_update_ctas(const PrbView& v, uint32_t b)
{
    // Many wide child groups per level (fanout 32, hundreds of entries) are more L2 misses than
    // one SM keeps in flight: then eight CTAs of one cluster share each level.
    return (v.fanout * b >= 8192u) ? 8u : 1u;
}

int prb_launch_update(const PrbView& v, uint32_t B, const int32_t* d_idx, const float* d_val, int raw,
                      float alpha, float eps, cudaStream_t s, uint32_t stale, bool linked)
{
    if (raw != 2) {
        if (prb_update_is_wide(v, B, false)) {
            const int k = prb_launch_update_wide(v, B, d_idx, d_val, raw, alpha, eps, s, stale);
            if (k != 0) return k;
        }
        PrbTreeArgs t;
        t.B = B; t.idx = d_idx; t.val = d_val; t.raw = raw; t.alpha = alpha; t.eps = eps; t.stale = stale;
        if (linked && B <= kPrbTreeEntries) t.most_ctas = 4u;      // (see prb_launch_insert)
        return prb_launch_tree(v, t, s, true);
    }
    static bool big_smem[kPrbMaxDevices];
    const int dev = prb_current_device();
    if (!big_smem[dev]) {
        const int most = (int)(prb_update_smem_bytes(PEARL_UPDATE_SUBBATCH) + 2 * kPrbTopFloats * sizeof(float));
        if (cudaFuncSetAttribute(prb_delta_kernel<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess ||
            cudaFuncSetAttribute(prb_delta_kernel<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess ||
            cudaFuncSetAttribute(prb_delta_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess ||
            cudaFuncSetAttribute(prb_delta_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess)
            return -1;
        big_smem[dev] = true;
    }
    // A batch beyond one CTA's reach goes sub-batch by sub-batch in batch order: every launch leaves
    // a consistent tree and later entries add to earlier ones, as in the whole batch.
    int launches = 0;
    for (uint32_t first = 0; first < B; first += PEARL_UPDATE_SUBBATCH) {
        const uint32_t b = B - first < PEARL_UPDATE_SUBBATCH ? B - first : PEARL_UPDATE_SUBBATCH;
        const uint32_t n2 = prb_update_n2(b);
        const uint32_t threads = n2 < 64 ? 64 : (n2 > 1024 ? 1024 : n2);
        const uint32_t ctas = prb_update_ctas(v, b);
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = prb_update_smem_bytes(n2) + v.top_floats * sizeof(float) * (v.min_off ? 2 : 1);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = ctas;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cudaError_t e = cudaSuccess;
#define PRB_LAUNCH_DELTA_AS(FF, MM) e = cudaLaunchKernelEx(&cfg, prb_delta_kernel<FF, MM>, v, b, n2, d_idx + first, d_val + first)
        PRB_WITH_TREE_OPTIONS(v, PRB_LAUNCH_DELTA_AS);
#undef PRB_LAUNCH_DELTA_AS
        if (e != cudaSuccess) return -1;
        ++launches;
    }
    return launches;
}
