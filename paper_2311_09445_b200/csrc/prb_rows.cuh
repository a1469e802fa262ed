// Short rows as words: the copy between the Data Storage (slots) and a dense batch, in either direction, without
// an index being divided.  A transition is numbered in words of 4 bytes (2 or 1 where a field's granule is
// smaller) over all its fields; a lane's word is fixed, so where it lies in a slot and in a row of the batch is
// looked up once, and consecutive lanes touch consecutive words.
#pragma once
#include "prb_internal.cuh"

// One field of the row: words of 2^log2 bytes, numbered from `first` over all fields.
struct PrbWordField {
    unsigned char* store;         // slot 0
    unsigned char* batch;         // row 0 of the batch
    uint32_t first, log2;
    uint32_t store_pitch, batch_pitch;
};
struct PrbWords {
    uint32_t n_words, chunks, lane_words;      // chunks of 32 words; lanes that share a row (8, 16 or 32)
    PrbWordField field[PRB_NUM_FIELDS];
};

inline PrbWords prb_plan_words(const PrbView& v, const PrbBatch& batch)
{
    PrbWords p;
    uint32_t words = 0;
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) {
        PrbWordField& fd = p.field[f];
        fd = PrbWordField{nullptr, nullptr, 0xFFFFFFFFu, 0u, 0u, 0u};
        if (batch.ptr[f] == nullptr || v.field_bytes[f] == 0) continue;
        fd.store = v.store[f];
        fd.batch = batch.ptr[f];
        fd.log2 = v.field_vec[f] >= 4u ? 2u : v.field_vec[f] == 2u ? 1u : 0u;
        fd.first = words;
        fd.store_pitch = v.field_pitch[f];
        fd.batch_pitch = v.field_bytes[f];
        words += v.field_bytes[f] >> fd.log2;
    }
    p.n_words = words;
    p.chunks = words ? (words + 31u) / 32u : 1u;
    p.lane_words = words <= 8u ? 8u : words <= 16u ? 16u : 32u;
    return p;
}

#ifdef __CUDACC__

struct PrbWord {
    unsigned char* store;
    unsigned char* batch;
    uint32_t store_pitch, batch_pitch, log2;
};
__device__ __forceinline__ PrbWord prb_find_word(const PrbWords& p, uint32_t w)
{
    PrbWord o = PrbWord{nullptr, nullptr, 0u, 0u, 0u};
#pragma unroll
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) {
        const PrbWordField& fd = p.field[f];
        if (w >= fd.first) {
            o.log2 = fd.log2; o.store_pitch = fd.store_pitch; o.batch_pitch = fd.batch_pitch;
            o.store = fd.store + ((uint64_t)(w - fd.first) << fd.log2);
            o.batch = fd.batch + ((uint64_t)(w - fd.first) << fd.log2);
        }
    }
    return o;
}

// The `warps` copying warps of a CTA share the rows: a warp takes a chunk of 32 words (or, with short rows, a whole
// row per `lane_words` lanes) and every `groups`-th of the CTA's rows; `first` is where the first chunk's word lies,
// looked up ahead of time.
struct PrbWordShare {
    uint32_t chunk, grp, groups;
    PrbWord first;
};
__device__ __forceinline__ PrbWordShare prb_word_share(const PrbWords& p, uint32_t warp, uint32_t warps)
{
    PrbWordShare g;
    g.groups = warps > p.chunks ? warps / p.chunks : 1u;
    g.grp = warp / p.chunks;
    g.chunk = warp - g.grp * p.chunks;
    if (g.grp >= g.groups) g.chunk = p.chunks;              // (a warp left over)
    g.first = prb_find_word(p, g.chunk * 32u + (threadIdx.x & (p.lane_words - 1u)));
    return g;
}

// Rows [k0, k0 + n) of the batch: up to eight loads of a thread in flight.  slot_of(r): the slot of row k0 + r.
template <bool kToStore, typename SlotOf>
__device__ __forceinline__ void prb_copy_words(const PrbWords& p, const PrbWordShare& g, uint32_t warps, uint32_t k0, uint32_t n, SlotOf slot_of)
{
    const uint32_t lane = threadIdx.x & 31u, per_row = p.lane_words, at_once = 32u / per_row;
    const uint32_t stride = g.groups * at_once, r_first = g.grp * at_once + lane / per_row;
    PrbWord o = g.first;
    for (uint32_t c = g.chunk; c < p.chunks; c += warps) {
        const uint32_t w = c * 32u + (lane & (per_row - 1u));
        if (c != g.chunk) o = prb_find_word(p, w);
        if (w >= p.n_words) continue;
        unsigned char* const batch = o.batch + (uint64_t)k0 * o.batch_pitch;
        constexpr int U = 8;
        for (uint32_t r0 = r_first; r0 < n; r0 += stride * U) {
            uint32_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t r = r0 + u * stride;
                if (r < n) {
                    const unsigned char* at = kToStore ? batch + (uint64_t)r * o.batch_pitch : o.store + (uint64_t)slot_of(r) * o.store_pitch;
                    if (o.log2 == 2u) v[u] = *reinterpret_cast<const uint32_t*>(at);
                    else if (o.log2 == 1u) v[u] = *reinterpret_cast<const uint16_t*>(at);
                    else v[u] = *at;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t r = r0 + u * stride;
                if (r < n) {
                    unsigned char* at = kToStore ? o.store + (uint64_t)slot_of(r) * o.store_pitch : batch + (uint64_t)r * o.batch_pitch;
                    if (o.log2 == 2u) *reinterpret_cast<uint32_t*>(at) = v[u];
                    else if (o.log2 == 1u) *reinterpret_cast<uint16_t*>(at) = (uint16_t)v[u];
                    else *at = (unsigned char)v[u];
                }
            }
        }
    }
}

// The same copy to the store, all n rows of a batch that lies in mapped host memory: 32 consecutive words of one field
// at a time, whatever rows they belong to, so that the link carries whole sectors (row by row, a sector of rewards
// or done bytes crossed it once per row).  256 rows of 165 bytes: 43.3 -> 41.2 us a step through host buffers.  `warp` of `warps` over all copying CTAs; four loads of a thread in flight.
template <typename SlotOf>
__device__ __forceinline__ void prb_copy_flat(const PrbWords& p, uint32_t warp, uint32_t warps, uint32_t n, SlotOf slot_of)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t total = 0;
#pragma unroll
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) if (p.field[f].batch) total += (n * (p.field[f].batch_pitch >> p.field[f].log2) + 31u) / 32u;
    constexpr int U = 4;
    for (uint32_t c0 = warp; c0 < total; c0 += warps * U) {
        uint32_t v[U], lg[U], at[U], pitch[U], row[U];
        unsigned char* store[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint32_t c = c0 + u * warps;
            store[u] = nullptr;
            v[u] = 0u;
            if (c >= total) continue;
#pragma unroll 1
            for (int f = 0; f < PRB_NUM_FIELDS; ++f) {
                const PrbWordField& fd = p.field[f];
                if (!fd.batch) continue;
                const uint32_t W = fd.batch_pitch >> fd.log2, words = n * W, here = (words + 31u) / 32u;
                if (c >= here) { c -= here; continue; }
                const uint32_t e = c * 32u + lane;
                if (e < words) {
                    row[u] = e / W; at[u] = (e - row[u] * W) << fd.log2; lg[u] = fd.log2; pitch[u] = fd.store_pitch; store[u] = fd.store;
                    const unsigned char* from = fd.batch + ((uint64_t)e << fd.log2);
                    v[u] = fd.log2 == 2u ? *reinterpret_cast<const uint32_t*>(from) : fd.log2 == 1u ? *reinterpret_cast<const uint16_t*>(from) : *from;
                }
                break;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (store[u] == nullptr) continue;
            unsigned char* to = store[u] + (uint64_t)slot_of(row[u]) * pitch[u] + at[u];
            if (lg[u] == 2u) *reinterpret_cast<uint32_t*>(to) = v[u];
            else if (lg[u] == 1u) *reinterpret_cast<uint16_t*>(to) = (uint16_t)v[u];
            else *to = (unsigned char)v[u];
        }
    }
}

#endif  // __CUDACC__
