// Single-pass decoupled look-back over per-tile status words: how a tile learns where its changed
// exponents start in its unit's payload (the sum of the payload bytes of the unit's earlier tiles)
// without a second pass.  Shared by the two sender kernels.
//
// Every wait is bounded: after kMaxPolls reads of a status word the waiting warp gives up, raises
// CIERA_ERR_TIMEOUT and carries on with offset 0 (output unspecified) instead of hanging.
#pragma once

#include "ciera_internal.cuh"

namespace ciera {

__device__ __forceinline__ unsigned long long ld_status(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_status(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Polls a tile status word until its flag is set.  Bounded: after max_polls reads (kMaxPolls in the
// kernels; the self-test passes a few dozen) it gives up, raises CIERA_ERR_TIMEOUT and returns
// "prefix 0" so that the caller finishes (with unspecified output) instead of hanging.
__device__ __forceinline__ unsigned long long wait_status(const unsigned long long* p, int32_t* status,
                                                          uint32_t max_polls = kMaxPolls) {
    unsigned long long st = ld_status(p);
    uint32_t polls = 0;
    while ((st >> 62) == 0) {
        if (++polls > max_polls) {
            if (status) atomicCAS(status, 0, (int32_t)CIERA_ERR_TIMEOUT);
            return kFlagPrefix;
        }
        if (polls > 16) __nanosleep(polls > 1024 ? 400 : 40);
        st = ld_status(p);
    }
    return st;
}

__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The short words and the groups of the whole step on long units (see ciera_internal.cuh).
__device__ __forceinline__ uint32_t ld_status(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_status(uint32_t* p, uint32_t v) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void add_status(unsigned long long* p, unsigned long long v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
// As wait_status (`st`: what was read last).
__device__ __forceinline__ uint32_t wait_status(const uint32_t* p, uint32_t st, int32_t* status) {
    uint32_t polls = 0;
    while ((st >> 30) == 0) {
        if (++polls > kMaxPolls) {
            if (status) atomicCAS(status, 0, (int32_t)CIERA_ERR_TIMEOUT);
            return kShortPrefix;
        }
        if (polls > 16) __nanosleep(polls > 1024 ? 400 : 40);
        st = ld_status(p);
    }
    return st;
}
__device__ __forceinline__ uint32_t wait_status(const uint32_t* p, int32_t* status) { return wait_status(p, ld_status(p), status); }

// A spread tile's payload bytes for the tiles behind it: its own status word and, where its group of 32 lies inside its
// unit, its group's (one thread).
__device__ __forceinline__ void report_tile(uint32_t* tile_status, unsigned long long* groups, const TileDesc& td, uint32_t tile,
                                            uint32_t bits, uint32_t bytes) {
    st_status(tile_status + tile, kShortAggregate | (bits << kShortBitsShift) | bytes);
    const uint32_t head = tile & ~(kGroupTiles - 1u);
    if (head >= td.first_tile && head + kGroupTiles - td.first_tile <= td.n_tiles_unit)
        add_status(groups + (tile >> kGroupTilesLog2), (1ull << kGroupCountShift) | bytes);
}

// Empties the status words of the tiles [lo, hi) and of their groups (thread `me` of n).
template <class WORD>
__device__ __forceinline__ void clear_status(WORD* tile_status, unsigned long long* groups, uint32_t lo, uint32_t hi, uint32_t me,
                                             uint32_t n) {
    for (uint32_t t = lo + me; t < hi; t += n) st_status(tile_status + t, (WORD)0);
    if (sizeof(WORD) == 8) return;  // no groups
    for (uint32_t g = (lo >> kGroupTilesLog2) + me; g < hi >> kGroupTilesLog2; g += n) st_status(groups + g, 0ull);
}

// Payload bytes of the unit's tiles before `tile` (one warp; first < tile): the words of the group that the tile is in, the
// words of the groups before it back to one that knows its prefix, and, where it comes to that, the words between
// the unit's first tile and its first whole group.  Tile words and the nearest 32 groups are fetched at once, so that the
// hundreds of tiles in work cost one round trip, where a word per tile, 32 to a round trip, took up to nine.  The last tile
// of a group adds the prefix to the group's word.
__device__ __forceinline__ uint64_t look_back(const uint32_t* tile_status, unsigned long long* groups, uint32_t first, uint32_t tile,
                                              int32_t* status, uint32_t lane) {
    const uint32_t head = tile & ~(kGroupTiles - 1u);
    const uint32_t whole = (first + kGroupTiles - 1u) & ~(kGroupTiles - 1u);  // the unit's first whole group starts here
    const bool near = tile - first <= kGroupTiles;  // the words before the tile reach back to the unit's start
    const uint32_t lo = near ? first : head;        // words [lo, tile), at most 32
    const uint32_t far_end = near ? first : whole;  // words [first, far_end), fewer than 32
    const bool has_near = lo + lane < tile, has_far = first + lane < far_end;
    uint32_t a = 0, c = 0;
    if (has_near) a = ld_status(tile_status + lo + lane);
    if (has_far) c = ld_status(tile_status + first + lane);
    // (32 bits hold it: a prefix lies at most as many groups back as can be in work, some 150 of 2^18 bytes)
    uint32_t sum = 0;
    uint64_t prefix = 0;
    bool from_start = true;  // no prefix was found: the words between first and far_end count
    if (!near) {
        const uint32_t g_first = whole >> kGroupTilesLog2;
        for (uint32_t g = head >> kGroupTilesLog2; g > g_first; g -= min(32u, g - g_first)) {
            const bool has = g_first + lane < g;  // lane l: the l-th group before group g
            const unsigned long long* const p = groups + (g - 1u - (has ? lane : 0u));
            unsigned long long st = has ? ld_status(p) : 0ull;
            uint32_t polls = 0, known;
            for (;;) {
                const bool ready = !has || ((st >> kGroupCountShift) & 63ull) == (unsigned long long)kGroupTiles;
                known = __ballot_sync(0xffffffffu, ready && (st >> 62) == 2ull);
                const uint32_t needed = known ? (known & (0u - known)) - 1u : 0xffffffffu;  // lanes below the nearest prefix
                if ((__ballot_sync(0xffffffffu, !ready) & needed) == 0u) break;
                if (++polls > kMaxPolls) {
                    if (status && lane == 0) atomicCAS(status, 0, (int32_t)CIERA_ERR_TIMEOUT);
                    known = 1u;
                    st = kFlagPrefix;
                    break;
                }
                if (polls > 16) __nanosleep(polls > 1024 ? 400 : 40);
                if (!ready) st = ld_status(p);
            }
            const uint32_t at = known ? (uint32_t)__ffs(known) - 1u : 32u;
            if (lane < at) sum += (uint32_t)(st & kValueMask);
            if (known) {
                prefix = __shfl_sync(0xffffffffu, st & kValueMask, (int)at);
                from_start = false;
                break;
            }
        }
    }
    uint32_t near_sum = 0;
    if (has_near) near_sum = wait_status(tile_status + lo + lane, a, status) & kShortValueMask;
    if (has_far && from_start) sum += wait_status(tile_status + first + lane, c, status) & kShortValueMask;
    __syncwarp();
    const uint64_t excl = prefix + __reduce_add_sync(0xffffffffu, sum) + __reduce_add_sync(0xffffffffu, near_sum);
    if (head >= first && tile - head == kGroupTiles - 1u) {
        const uint64_t before_group = excl - __reduce_add_sync(0xffffffffu, lo + lane >= head ? near_sum : 0u);
        if (lane == 0) add_status(groups + (head >> kGroupTilesLog2), kFlagPrefix + before_group);
    }
    return excl;
}

// One byte of a message; with TWICE also `twin` bytes further on (the whole-step kernel writes a message into the
// sender's and the receiver's buffer alike).
template <bool TWICE>
__device__ __forceinline__ void put_byte(uint8_t* p, uint8_t v, int64_t twin) {
    p[0] = v;
    if (TWICE) p[twin] = v;
}

// The unit's last tile reports the totals and zeroes the two pads (one warp).
template <int DT, bool TWICE>
__device__ __forceinline__ void finish_unit(const TileDesc& td, uint32_t log2b, uint64_t total, uint8_t* msgs, int64_t twin,
                                            unsigned long long* wire_bytes, uint32_t* changed_blocks, uint32_t lane) {
    const uint64_t N = td.n_unit;
    uint8_t* msg = msgs + td.msg_off;
    const uint64_t smoff = sm_offset(N, log2b);
    const uint64_t sm_bytes = sm_section_bytes(N, DT);
    const uint64_t payoff = smoff + pad16(sm_bytes);
    if (lane == 0) {
        wire_bytes[td.unit] = payoff + total;
        // every changed block carries a full block's bytes except possibly the last one, which carries fewer
        if (DT == CIERA_FP16) {
            const uint64_t bpb = payload_bytes_of_blocks<DT>(1, log2b);
            changed_blocks[td.unit] = (uint32_t)((total + bpb - 1u) / bpb);
        } else {
            changed_blocks[td.unit] = (uint32_t)((total + (1ull << log2b) - 1u) >> log2b);
        }
    }
    for (uint64_t b = bitmap_bytes(N, log2b) + lane; b < smoff; b += 32) put_byte<TWICE>(msg + b, 0, twin);
    for (uint64_t b = smoff + sm_bytes + lane; b < payoff; b += 32) put_byte<TWICE>(msg + b, 0, twin);
}

// Resolver warp, one spread tile: exclusive prefix of the payload bytes over the earlier tiles of
// the same unit by a single-pass look-back over the status words, then the duties that need it.
// (WORD: short words and groups, or one 64-bit word per tile.)
// `known` is called with the tile's exclusive payload offset inside its unit as soon as there is one (the tile's flags
// in `bm` are not read after that).
template <int DT, bool TWICE, class WORD, class KNOWN>
__device__ __forceinline__ void resolve_tile(const TileDesc& td, uint32_t tile, uint32_t log2b, uint64_t agg,
                                                 const uint32_t* bm, uint8_t* msgs, int64_t twin,
                                                 unsigned long long* wire_bytes, uint32_t* changed_blocks, WORD* tile_status,
                                                 unsigned long long* groups, int32_t* status, uint32_t lane, KNOWN known) {
    constexpr bool kShort = sizeof(WORD) == 4;
    const uint32_t nbt = kTileValues >> log2b;
    uint8_t* msg = msgs + td.msg_off;
    const uint32_t mybits = nbt < 8 ? bm[0] : 0u;

    uint64_t excl = 0;
    if constexpr (kShort) {
        if (td.tile_in_unit != 0) excl = look_back(tile_status, groups, td.first_tile, tile, status, lane);
    } else if (td.tile_in_unit != 0) {
        int64_t hi = (int64_t)tile - 1;
        while (true) {
            const int64_t idx = hi - (int64_t)lane;
            unsigned long long st = kFlagPrefix;  // "prefix 0" stands before the unit's first tile
            if (idx >= (int64_t)td.first_tile) st = wait_status(tile_status + idx, status);
            __syncwarp();
            const uint32_t pmask = __ballot_sync(0xffffffffu, (st >> 62) == 2ull);
            const uint32_t first = pmask ? (uint32_t)__ffs(pmask) - 1u : 31u;
            excl += warp_sum_u64(lane <= first ? (st & kValueMask) : 0ull);
            if (pmask) break;
            hi -= 32;
        }
        if (lane == 0)
            st_status(tile_status + tile, kFlagPrefix | ((unsigned long long)mybits << kBitsShift) | (excl + agg));
    }
    __syncwarp();  // every lane has read its flags
    known(excl);

    // tiles of fewer than 8 blocks share a bitmap byte: the last tile of each byte collects the
    // bits its predecessors published in their status words
    if (nbt < 8) {
        const uint32_t tpb = 8u / nbt;
        const uint32_t p = td.tile_in_unit & (tpb - 1u);
        if (p == tpb - 1u || td.tile_in_unit == td.n_tiles_unit - 1u) {
            uint32_t part = 0;
            if (lane < p) {
                const auto st = wait_status(tile_status + (tile - p + lane), status);
                part = (uint32_t)((st >> (kShort ? kShortBitsShift : kBitsShift)) & 0x3Fu) << (lane * nbt);
            }
            __syncwarp();
            part = __reduce_or_sync(0xffffffffu, part);
            if (lane == 0) put_byte<TWICE>(msg + td.tile_in_unit / tpb, (uint8_t)(part | (mybits << (p * nbt))), twin);
        }
    }
    if (td.tile_in_unit == td.n_tiles_unit - 1u)
        finish_unit<DT, TWICE>(td, log2b, excl + agg, msgs, twin, wire_bytes, changed_blocks, lane);
}

}  // namespace ciera
