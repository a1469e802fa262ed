// The copy of rows between the Data Storage (slots) and a dense batch, through registers, in three ways.
//
// Words (rows of up to kPrbMostWords of them): no index is divided.  A transition is numbered in words of 4 bytes (2 or 1
// where a field's granule is smaller) over all its fields; a lane's word is fixed, so where it lies in a slot and in a row of
// the batch is looked up once, and consecutive lanes touch consecutive words.
// Tiles (an insertion's longer rows): kPrbTile consecutive granules (the largest power of two up to 16 bytes that divides
// the field) of one field, whatever rows they belong to; a division each.  A row is no unit of work, so one long row keeps
// several CTAs busy and a thread moves up to 16 bytes at a time.
// Units (a sample's longer rows): all the granules of a CTA's rows, field by field, dealt to its threads; a division each,
// loads of several fields in flight at once.
// us a call, as words / this way: insertion of 1 row of 14 KB 9.4 / 3.8, of 256 11.2 / 4.4, of one row of 56 KB of an odd size
// 131 / 3.6; sample of 512 rows of 2 KB 19 / 7.0, of 8 KB 46 / 10, of 64 rows of 56 KB of an odd size 141 / 60.
#pragma once
#include "prb_internal.cuh"

// One field of the row: words of 2^log2 bytes, numbered from `first` over all fields.
struct PrbWordField {
    unsigned char* store;         // slot 0
    unsigned char* batch;         // row 0 of the batch
    uint32_t first;
    uint16_t log2, unit;                       // log2 of the word and of the granule (few bytes: a cold line of parameters is 84 cycles)
    uint32_t store_pitch, batch_pitch;
    PRB_HD uint32_t units() const { return batch_pitch >> unit; }      // granules per row
};
struct PrbWords {
    uint32_t n_words, chunks, lane_words;      // chunks of 32 words; lanes that share a row (8, 16 or 32)
    uint32_t units;                            // granules per row over all fields; 0: too many of them for 32 bits
    uint32_t fine;                             // 1: most of the row is granules of up to 4 bytes (and all of it is copied as such)
    PrbWordField field[PRB_NUM_FIELDS];
};
constexpr uint32_t kPrbMostWords = 64;
constexpr uint32_t kPrbTile = 2048;

inline PrbWords prb_plan_words(const PrbView& v, const PrbBatch& batch)
{
    PrbWords p;
    uint32_t words = 0, coarse = 0;
    uint64_t units = 0;
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) {
        PrbWordField& fd = p.field[f];
        fd = PrbWordField{nullptr, nullptr, 0xFFFFFFFFu, 0, 0, 0u, 0u};
        if (batch.ptr[f] == nullptr || v.field_bytes[f] == 0) continue;
        fd.store = v.store[f];
        fd.batch = batch.ptr[f];
        fd.log2 = (uint16_t)(v.field_vec[f] >= 4u ? 2u : v.field_vec[f] == 2u ? 1u : 0u);
        fd.first = words;
        fd.store_pitch = v.field_pitch[f];
        fd.batch_pitch = v.field_bytes[f];
        words += v.field_bytes[f] >> fd.log2;
        while ((1u << fd.unit) < v.field_vec[f]) ++fd.unit;
        units += v.field_bytes[f] >> fd.unit;
        if (fd.unit > 2u) coarse += v.field_bytes[f] >> fd.log2;
    }
    p.fine = coarse < words - coarse ? 1u : 0u;
    if (p.fine) {
        // (then the other fields go as units of 4 bytes, too)
        for (int f = 0; f < PRB_NUM_FIELDS; ++f) {
            PrbWordField& fd = p.field[f];
            if (fd.unit <= 2u) continue;
            units += ((uint64_t)fd.units() << (fd.unit - 2u)) - fd.units();
            fd.unit = 2u;
        }
    }
    p.units = units * v.max_batch < (1ull << 31) ? (uint32_t)units : 0u;
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

// Tile `tile` of the n rows of a batch, to the store, by the whole CTA.
template <typename T, typename SlotOf>
__device__ __forceinline__ void prb_copy_tile(const PrbWordField& fd, uint32_t n, uint32_t tile, SlotOf slot_of)
{
    const uint32_t W = fd.units(), e0 = tile * kPrbTile, e1 = (uint32_t)min((uint64_t)n * W, (uint64_t)e0 + kPrbTile);      // (n W is below 2^32)
    const uint64_t Wp = fd.store_pitch / sizeof(T);
    prb_copy_mapped<T>(reinterpret_cast<T*>(fd.store), reinterpret_cast<const T*>(fd.batch), e0, e1, [](uint32_t e) { return (uint64_t)e; },
                       [=](uint32_t e) { const uint32_t r = e / W; return (uint64_t)slot_of(r) * Wp + (e - r * W); }, threadIdx.x, blockDim.x);
}
// All tiles, shared out over `ctas` CTAs of which this one is number `cta`.
template <typename SlotOf>
__device__ __forceinline__ void prb_copy_tiles(const PrbWords& p, uint32_t cta, uint32_t ctas, uint32_t n, SlotOf slot_of)
{
    auto tiles = [&](int f) { return (uint32_t)(((uint64_t)n * p.field[f].units() + kPrbTile - 1u) / kPrbTile); };
    uint32_t total = 0;
#pragma unroll
    for (int f = 0; f < PRB_NUM_FIELDS; ++f) total += tiles(f);
    const uint32_t t_lo = (uint32_t)(((uint64_t)cta * total) / ctas), t_hi = (uint32_t)(((uint64_t)(cta + 1u) * total) / ctas);
    for (uint32_t t = t_lo; t < t_hi; ++t) {
        uint32_t tile = t;
        int f = 0;
        for (; f + 1 < PRB_NUM_FIELDS; ++f) {
            const uint32_t here = tiles(f);
            if (tile < here) break;
            tile -= here;
        }
        const PrbWordField& fd = p.field[f];
        switch (fd.unit) {
        case 4: prb_copy_tile<uint4>(fd, n, tile, slot_of); break;
        case 3: prb_copy_tile<uint2>(fd, n, tile, slot_of); break;
        case 2: prb_copy_tile<uint32_t>(fd, n, tile, slot_of); break;
        case 1: prb_copy_tile<uint16_t>(fd, n, tile, slot_of); break;
        default: prb_copy_tile<unsigned char>(fd, n, tile, slot_of); break;
        }
    }
}

// Rows [k0, k0 + n) of the batch as units, from the store, by `nthreads` threads of which this one has rank `rank`; four loads of
// a thread in flight.
template <typename SlotOf>
__device__ __forceinline__ void prb_copy_units(const PrbWords& p, uint32_t rank, uint32_t nthreads, uint32_t k0, uint32_t n, SlotOf slot_of)
{
    constexpr int U = 4;
    const uint32_t total = p.units * n;
    for (uint32_t e0 = rank; e0 < total; e0 += nthreads * U) {
        uint4 v[U];
        unsigned char* to[U];
        uint32_t lg[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint32_t e = e0 + u * nthreads;
            to[u] = nullptr;
            lg[u] = 0u;
            v[u] = make_uint4(0u, 0u, 0u, 0u);
            if (e >= total) continue;
            int f = 0;
#pragma unroll
            for (int g = 0; g + 1 < PRB_NUM_FIELDS; ++g) {
                const uint32_t here = p.field[g].units() * n;
                if (f == g && e >= here) { e -= here; f = g + 1; }
            }
            const PrbWordField& fd = p.field[f];
            const uint32_t W = fd.units(), r = e / W, at = (e - r * W) << fd.unit;
            const unsigned char* const from = fd.store + (uint64_t)slot_of(r) * fd.store_pitch + at;
            to[u] = fd.batch + (uint64_t)(k0 + r) * fd.batch_pitch + at;
            lg[u] = fd.unit;
            switch (fd.unit) {
            case 4: v[u] = *reinterpret_cast<const uint4*>(from); break;
            case 3: { const uint2 t = *reinterpret_cast<const uint2*>(from); v[u].x = t.x; v[u].y = t.y; break; }
            case 2: v[u].x = *reinterpret_cast<const uint32_t*>(from); break;
            case 1: v[u].x = *reinterpret_cast<const uint16_t*>(from); break;
            default: v[u].x = *from; break;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (to[u] == nullptr) continue;
            switch (lg[u]) {
            case 4: *reinterpret_cast<uint4*>(to[u]) = v[u]; break;
            case 3: *reinterpret_cast<uint2*>(to[u]) = make_uint2(v[u].x, v[u].y); break;
            case 2: *reinterpret_cast<uint32_t*>(to[u]) = v[u].x; break;
            case 1: *reinterpret_cast<uint16_t*>(to[u]) = (uint16_t)v[u].x; break;
            default: *to[u] = (unsigned char)v[u].x; break;
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
