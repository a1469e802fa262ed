// Index arithmetic of the tree work that holds on host and device alike (and is tested on the host).
#pragma once
#include <stdint.h>
#ifdef __CUDACC__
#define PRB_HD __host__ __device__ __forceinline__
#else
#define PRB_HD inline
#endif

// Nodes of a level whose nodes cover 2^shift leaves each, over `capacity` (1 .. 2^30) leaves.  The shift of the root's
// level may be 32 (fanout 16 above 2^28 slots); a 32-bit value is not shifted by that much.
PRB_HD uint32_t prb_nodes_covering(uint32_t capacity, uint32_t shift)
{
    return ((capacity - 1u) >> (shift < 31u ? shift : 31u)) + 1u;
}
