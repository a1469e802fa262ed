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

// Where index i starts in a hash table of 2^(32 - shift) places: the high bits of the product, which every bit of the index
// reaches (its middle bits are the same for all multiples of a large power of two -- the heads of parallel segments of a
// ring, say -- which then probed one after another: up to 1024 shared atomics in a line).
PRB_HD uint32_t prb_hash_place(uint32_t i, uint32_t shift) { return (i * 0x9E3779B1u) >> shift; }
