// Internal declarations shared by the translation units of libciera (not installed).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <vector>

#include "ciera.h"

namespace ciera {

// One tile = kTileValues consecutive values of one unit = the work of one thread block.
// Each thread owns kVPT consecutive values ("a group"): 16 values are 16 exponent bytes, i.e.
// one 128-bit access on each of the byte-wide streams (cache, sm, payload).
constexpr int kThreads = 512;
constexpr int kVPT = 16;
constexpr int kTileValues = kThreads * kVPT;  // 8192
constexpr int kWarps = kThreads / 32;
// Block sizes come in two classes.  "Coarse" blocks (16 values and more) hold whole pieces, so a
// piece has one flag and a tile at most 512 blocks; "fine" blocks (1, 2, 4 or 8 values) are
// smaller than (or as large as) a piece, a piece has several flags and a tile up to 8192 blocks.
constexpr uint32_t kFineLog2 = 4;                    // log2b < kFineLog2: fine
constexpr int kBitmapWords = kTileValues / 16 / 32;  // 16: words of block flags of a tile, coarse
constexpr int kFineBitmapWords = kTileValues / 32;   // 256: the same, fine
__host__ __device__ inline bool is_fine(uint32_t log2b) { return log2b < kFineLog2; }

constexpr uint32_t kNoTile = 0xffffffffu;

// Device-side tile descriptor: everything a thread block needs, in one 48-byte record so that
// a single dependent load stands between block start and the first data load.
struct __align__(16) TileDesc {
    uint64_t w_off;         // byte offset of the tile's first value in the weights buffer
    uint64_t c_off;         // byte offset of the tile's first value in the cache
    uint64_t msg_off;       // byte offset of the unit's message slot
    uint64_t n_unit;        // N of the unit
    uint32_t unit;          // index into the per-unit outputs
    uint32_t tile_in_unit;  // 0 .. n_tiles_unit-1
    uint32_t first_tile;    // table index of the unit's first tile
    uint32_t n_tiles_unit;  // tiles of this unit
};
static_assert(sizeof(TileDesc) == 48, "TileDesc must stay three 16-byte words");

// Tile status word used by the single-pass look-back of the encode kernel.
//   bits 63:62  0 = empty, 1 = aggregate of this tile, 2 = inclusive prefix up to this tile
//   bits 61:56  the tile's own bitmap bits when a tile holds fewer than 8 blocks
//   bits 55:0   payload bytes
constexpr unsigned long long kFlagAggregate = 1ull << 62;
constexpr unsigned long long kFlagPrefix = 2ull << 62;
constexpr unsigned long long kValueMask = (1ull << 56) - 1;
constexpr int kBitsShift = 56;

// The whole step on tables of long units (LONG in ciera_encode.cu) keeps shorter words per tile, and words per group of 32
// tiles that start at a multiple of 32 and belong to one unit.
//   tile   bits 31:30 as above, bits 29:24 the tile's own bitmap bits, bits 23:0 payload bytes of the tile (at most
//          kTileValues) or, handed on by a run, of its unit so far (at most kSeqMaxTiles times that)
//   group  bits 63:62 2 = the value goes back to the unit's first tile, bits 61:56 tiles that have reported, bits 55:0 payload
//          bytes; everything in it is added, in any order
constexpr uint32_t kShortAggregate = 1u << 30;
constexpr uint32_t kShortPrefix = 2u << 30;
constexpr uint32_t kShortValueMask = (1u << 24) - 1;
constexpr int kShortBitsShift = 24;
constexpr uint32_t kGroupTilesLog2 = 5, kGroupTiles = 1u << kGroupTilesLog2;
constexpr int kGroupCountShift = 56;

// Upper bound on polls of one status word before a tile gives up and raises CIERA_ERR_TIMEOUT.
constexpr uint32_t kMaxPolls = 1u << 21;

template <int DT>
struct Traits;
template <>
struct Traits<CIERA_BF16> {
    static constexpr int kValueBytes = 2;
    static constexpr int kSmBytes = 1;
};
template <>
struct Traits<CIERA_FP32> {
    static constexpr int kValueBytes = 4;
    static constexpr int kSmBytes = 3;
};
// fp16: 11 bits of sign-plus-mantissa and 5 exponent bits per value on the wire, so the byte
// counts below hold for multiples of 8 values only (kSmBytes is not used for it)
template <>
struct Traits<CIERA_FP16> {
    static constexpr int kValueBytes = 2;
    static constexpr int kSmBytes = 0;
};
// bytes of sign-plus-mantissa of `values` values (a multiple of 8 for fp16), and payload bytes of
// `blocks` full blocks
template <int DT>
__host__ __device__ constexpr uint64_t sm_bytes_of_values(uint64_t values) {
    return DT == CIERA_FP16 ? (values >> 3) * 11 : values * Traits<DT>::kSmBytes;
}
template <int DT>
__host__ __device__ constexpr uint64_t payload_bytes_of_blocks(uint64_t blocks, uint32_t log2b) {
    // fp16: five bits per exponent, a block rounded up to whole bytes (1, 2, 3, 5, 10, 20, ... bytes)
    return DT == CIERA_FP16 ? blocks * (((5ull << log2b) + 7ull) >> 3) : blocks << log2b;
}

__host__ __device__ inline uint64_t pad16(uint64_t x) { return (x + 15ull) & ~15ull; }
__host__ __device__ inline uint64_t num_blocks(uint64_t n, uint32_t log2b) {
    return (n + (1ull << log2b) - 1) >> log2b;
}
// Tiles per segment of a unit of n_tiles tiles whose changed blocks before each tile are counted ahead of decode
// (a power of two; at most 32 segments, so that one lane each can fetch their totals; a segment has work enough
// for one thread block of the prefix kernel: with fine blocks 128 bytes to 1 KB of flags per tile, else a few words)
__host__ __device__ inline uint32_t prefix_segment(uint32_t n_tiles, bool fine) {
    uint32_t s = fine ? 16u : 256u;
    while (32u * s < n_tiles) s *= 2u;
    return s;
}
__host__ __device__ inline uint64_t bitmap_bytes(uint64_t n, uint32_t log2b) { return (num_blocks(n, log2b) + 7) >> 3; }
__host__ __device__ inline uint64_t sm_offset(uint64_t n, uint32_t log2b) { return pad16(bitmap_bytes(n, log2b)); }
__host__ __device__ inline uint64_t payload_offset(uint64_t n, uint32_t sm_bytes_per_value, uint32_t log2b) {
    return sm_offset(n, log2b) + pad16(n * sm_bytes_per_value);
}

// The same sizes by precision, for code that also handles fp16 (5 exponent bits and 11
// sign-plus-mantissa bits per value, packed without gaps; every changed block of the payload starts
// on a byte boundary).
__host__ __device__ inline uint32_t sm_bits_of(int dtype) { return dtype == CIERA_FP32 ? 24u : dtype == CIERA_FP16 ? 11u : 8u; }
__host__ __device__ inline uint32_t exp_bits_of(int dtype) { return dtype == CIERA_FP16 ? 5u : 8u; }
__host__ __device__ inline uint64_t sm_section_bytes(uint64_t n, int dtype) { return (n * sm_bits_of(dtype) + 7) >> 3; }
__host__ __device__ inline uint64_t block_payload_bytes(uint64_t len, int dtype) { return (len * exp_bits_of(dtype) + 7) >> 3; }
__host__ __device__ inline uint64_t payload_offset_of(uint64_t n, int dtype, uint32_t log2b) {
    return sm_offset(n, log2b) + pad16(sm_section_bytes(n, dtype));
}
// the largest payload a unit of n values can have: every block changed
__host__ __device__ inline uint64_t payload_bytes_max(uint64_t n, int dtype, uint32_t log2b) {
    const uint64_t nb = num_blocks(n, log2b);
    if (nb == 0) return 0;
    return (nb - 1) * block_payload_bytes(1ull << log2b, dtype) + block_payload_bytes(n - ((nb - 1) << log2b), dtype);
}

// Units with more blocks than this get their per-tile "changed blocks before" counts from a
// prefix kernel at decode time; shorter ones read them straight from the bitmap.  With fine
// blocks every unit of more than one tile goes through the prefix kernel.
constexpr uint32_t kDecodeDirectBlocks = 4096;

// Layout of the scratch ("workspace") of a plan with nt tiles, shared by the sender, transport and receiver calls:
//   [0, 8 nt)             one 64-bit look-back status word per tile                     (sender)
//                         or, the whole step on long units: a 32-bit word per tile, then a 64-bit word per whole group
//   [8 nt, + 16)          the sender's counters of runs, of finished blocks and of spread tiles (sender)
//   [8 nt + 16, + 16)     the counter that transport and receiver hand their tiles out from, and their count of
//                         thread blocks (producer warps) that have drawn their last number
//   [8 nt + 32, + 4 nt)   changed blocks before each tile of the units that go through the receiver's prefix kernel
// Sender, transport and receiver each need their counters all zero when they start and leave them so (the last
// thread block to finish, or the last draw, clears them), so that no call needs a clearing launch in front of its kernel;
// transport and receiver touch nothing of the sender's, and the per-tile counts need no initial value.
__host__ __device__ inline size_t workspace_groups_offset(size_t nt) { return (nt * sizeof(uint32_t) + 7) / 8 * 8; }
__host__ __device__ inline size_t workspace_sender_counters_offset(size_t nt) { return nt * sizeof(unsigned long long); }
__host__ __device__ inline size_t workspace_ticket_offset(size_t nt) { return workspace_sender_counters_offset(nt) + 16; }
__host__ __device__ inline size_t workspace_prefix_offset(size_t nt) { return workspace_ticket_offset(nt) + 16; }
__host__ __device__ inline size_t workspace_total_bytes(size_t nt) {
    return (workspace_prefix_offset(nt) + nt * sizeof(uint32_t) + 15) / 16 * 16;
}

// Entropy stage: a unit of up to this many segment slots is coded by one thread block, a longer one by several.
constexpr uint32_t kEntLongSlots = 64;

// The tile table lists the tiles of "short" units (up to this many tiles) first, longest units
// first, then the tiles of the longer units.  The encode kernel lets one thread block work through
// a short unit tile after tile (the tile's place in the payload is then a running sum inside the
// block) and spreads everything else tile by tile over all blocks.
constexpr uint32_t kSeqMaxTiles = 32;
// Which tables a whole step with coarse blocks runs with the instance for long units.  Counted as long are the tiles of units of
// more than 32 tiles, in fp16 of more than 128, and there have to be kLongTilesMin of them: 8 to each of the 296 thread
// blocks of a B200, for with few tiles to a block the sending that is put off has nothing to hide behind.  One tensor on
// four shards, us by the other instance / by this one (fp32, of whose blocks there are 148, breaks even at 1500 tiles):
//   tiles   1448         2048         2435         4096           16384          32768
//   bf16    32.7 / 34.5  41.6 / 40.9  49.2 / 46.4  71.5 / 63.3    246 / 206      477 / 396
//   fp32    51.4 / 51.7  68.6 / 64.3  79.0 / 75.0  126.5 / 110.3  466 / 391
//   fp16    35.2 / 37.6  45.2 / 46.1  52.4 / 52.6  77.1 / 73.7    269 / 250      523 / 485
// bf16 and fp32 gain with every block size and rate of change from there on.  In fp16, whose consumers have the most to do to a
// tile, small tables of long units lose where much changes (seven units of 400 tiles 61.7 / 65.2, 24 of 190 94.9 / 98.6, 43 of
// 190 160.5 / 160.4), units of 34 to 100 tiles lose at any rate (240 of 34 133.5 / 139.4), and blocks of 32 and 64 values lose 3 to
// 6 % where most change and a few, scattered, do not, as much as they gain where few change (2^28 values, four units: blocks of 64
// 613.8 / 639.7 and 529.4 / 490.1; of 128 597.8 / 599.3, of 256 555.8 / 521.9; 28 units of 300 tiles, blocks of 16, 192.3 / 169.0).
// Parts of a host step take the instance that the whole step would, since their status words have to be the same; they
// have few tiles to a block, but wait for the link (2^25 bf16 values 1686 us by either, fp32 3196 and 3211 with runs 30 apart).
constexpr uint32_t kLongTilesMin = 8 * 296;
constexpr uint32_t kLongTilesMinFp16 = 8192;
inline uint32_t long_unit_tiles(int dtype) { return dtype == CIERA_FP16 ? 128u : kSeqMaxTiles; }
// Shorter units beside the long ones are slower by that instance where their tiles are not full, in fp16, and in fp32 with
// blocks of 16 values, so there have to be as many long tiles as the weight of these:
//                              lost by such a tile, ns        gained by a long tile, ns      weight
//   bf16 ragged                0.6 to 1.3                     2.0 to 2.5                     1
//   fp32 ragged                4.1 to 5.1                     3.9 to 4.6                     2
//   fp32 all, blocks of 16     5.2                            3.0                            2
//   fp16 full / ragged         0.3 to 0.95 / 0.9 to 8.8       0.8 to 1.1                     1 / 10
// Units of 1024 values from 12 288 tensors beside one tensor of 2^25, by the other instance / by this one: bf16 1299 / 1522 us,
// fp32 2026 / 3041, fp16 1869 / 2024; half an OLMoE-shaped layer beside 2^25, fp32 in blocks of 16, 676 / 790; a layer beside 2^25,
// bf16 631 / 625, fp16 in blocks of 64 680 / 706.
inline bool runs_as_long_units(int dtype, uint32_t log2b, uint64_t long_tiles, uint64_t other_tiles, uint64_t other_ragged) {
    if (dtype == CIERA_FP16)
        return log2b != 5 && log2b != 6 && long_tiles >= kLongTilesMinFp16 && long_tiles >= other_tiles + 9 * other_ragged;
    const uint64_t slow = dtype == CIERA_BF16 ? other_ragged : 2 * (log2b == 4 ? other_tiles : other_ragged);
    return long_tiles >= kLongTilesMin && long_tiles >= slow;
}
// That needs many more units than thread blocks: a table whose short units' tiles are fewer than kSpreadShare times
// the longest of these units would leave most of the GPU idle while a few blocks work through their units, so the
// encode kernel spreads all tiles of such a table.  197 = 2/3 of the 296 thread blocks that a B200
// holds, where the two ways cross.  Whole step, bf16, units of 16 tiles, in runs / spread: 64 tiles 26.4 / 7.7 us,
// 768 tiles 26.2 / 12.9, 2048 tiles 40.0 / 34.6, 3072 tiles 47.1 / 50.0, 49152 tiles 570 / 625; units of 32 tiles:
// 1536 tiles 50.4 / 23.5, 4096 tiles 76.5 / 63.0.  (Measured on the bf16 step, which has 296 blocks; the plan does not know
// which kernel will run.  The fp32 step has 148, so its ways cross at half as many tiles, which has not been measured; of 78
// tables in all precisions none is slower than with runs only, the hashed sender's included.)
constexpr uint32_t kSpreadShare = 197;
constexpr uint32_t kEncodeBlocks = 296;  // the encode kernel's thread blocks on a B200, two on each of 148 SMs
constexpr uint32_t kRunsPerBlock = 8;    // runs of short units to a block below which long runs are cut (ciera_plan_create)
// A short unit is handed out in runs of this many tiles (all units' first runs, then all second runs, ...): the
// smaller the piece of work a thread block draws, the less the blocks differ in when they finish.  A run's first
// tile takes its payload offset from the status word that the run before it left.  A multiple of 4, so that tiles
// sharing a bitmap byte (blocks of 2048 and 4096 values) stay in one run.
constexpr uint32_t kSeqRunTiles = 4;

// Bytes of a message slot that tile j of a unit moves in the transport kernel: [j * chunk,
// (j + 1) * chunk); the unit's last tile also moves whatever lies beyond (pads and, for coarse
// blocks, the bitmap: less than 100 bytes per unit plus one bitmap byte per 8 blocks).  With fine
// blocks the bitmap is a sizeable part of the message, so the chunk grows by a tile's share of it.
__host__ __device__ inline uint64_t transport_chunk_bytes(uint32_t sm_bytes_per_value, uint32_t log2b) {
    const uint64_t bitmap_share = is_fine(log2b) ? pad16((uint64_t)kTileValues >> (log2b + 3)) : 0;
    return (uint64_t)kTileValues * (sm_bytes_per_value + 1) + bitmap_share;
}

// the largest number of parts that a step on host weights is cut into
constexpr uint32_t kHostPartsMax = 64;

}  // namespace ciera

// The plan object behind the opaque handle.
struct ciera_plan {
    int dtype = 0;
    uint32_t block = 0;
    uint32_t log2b = 0;
    uint32_t n_units = 0;
    uint64_t total_values = 0;
    bool has_empty_units = false;
    std::vector<ciera_unit> units;
    std::vector<ciera::TileDesc> tiles;
    std::vector<uint32_t> prefix_segments;  // first tiles of the segments of every unit whose decode needs the prefix kernel
    bool prefix_segmented = false;          // one of these units has several segments
    std::vector<uint32_t> seq_first;   // first tile of every short unit, in table order, + end marker
    struct SeqRun {
        uint32_t lo, hi;               // tiles [lo, hi) of the table
    };
    bool long_units = false;           // a whole step with coarse blocks is run by the instance for long units
    bool spread_all = false;           // the short units' tiles are spread too (kSpreadShare)
    std::vector<SeqRun> seq_runs;      // the short units' runs of tiles in the order they are handed out
    std::vector<uint32_t> unit_first;  // first tile of every unit (0xffffffff: a unit without values)
    std::vector<uint64_t> hash_base;   // index of every unit's first block in a per-block hash cache
    std::vector<uint64_t> tile_hash;   // the same for every tile's first block, in tile-table order
    // the numbers of the tiles by ascending address of their weights, for steps on host weights; left empty where that
    // is the order of `tiles` already.  by_address_ok: the units' weights do not overlap.
    std::vector<uint32_t> tiles_by_address;
    bool by_address_ok = false;
    uint64_t total_blocks = 0;
    std::vector<uint64_t> seg_base;    // index of every unit's first 4096-byte payload segment (entropy stage)
    uint64_t total_segments = 0;
    // the ends of the units' furthest values and slots in the three kinds of buffers, in bytes
    uint64_t cache_extent = 0, weights_extent = 0, msg_extent = 0;
    // the tiles whose values, rounded up to 16 bytes, go past these ends (kNoTile: none; several: more than these)
    uint32_t weights_end_tile = ciera::kNoTile, cache_end_tile = ciera::kNoTile;
    bool several_end_tiles = false;
    // entropy stage: units of more than kEntLongSlots segment slots, and their chunks of as many
    // {unit, first segment of the chunk inside the unit, index among the long units, 0}
    struct EntChunk {
        uint32_t unit, first_seg, long_index, zero;
    };
    std::vector<uint32_t> ent_long_units;
    std::vector<EntChunk> ent_chunks;
    const uint32_t* ent_long_units_dev = nullptr;
    const uint4* ent_chunks_dev = nullptr;
    std::vector<uint8_t> image;        // device image: tiles, prefix_segments, seq_first, hash_base, unit_first, seg_base, units,
                                       // ent_long_units, ent_chunks, tiles_by_address, tile_hash, seq_runs
    const ciera::TileDesc* tiles_dev = nullptr;
    const uint32_t* tiles_by_address_dev = nullptr;
    const uint32_t* prefix_segments_dev = nullptr;
    const uint32_t* seq_first_dev = nullptr;
    const uint2* seq_runs_dev = nullptr;
    const unsigned long long* hash_base_dev = nullptr;
    const unsigned long long* tile_hash_dev = nullptr;
    const uint32_t* unit_first_dev = nullptr;
    const unsigned long long* seg_base_dev = nullptr;
    const ciera_unit* units_dev = nullptr;
};

namespace ciera {
int record_cuda_error(cudaError_t e);          // stores e for ciera_last_cuda_error, returns CIERA_ERR_CUDA
void count_launch();                           // launch accounting
// A launch that may begin while the kernel before it in the stream still drains (programmatic dependent launch): blocks
// become resident as soon as there is room, set themselves up and wait in pdl_wait() -- which every thread of such a
// kernel calls before it touches global memory -- until the kernel before has finished and its writes are visible.
// Only the tables of a plan's device image may be read earlier (the sender kernels do): ciera_plan_bind has waited for the
// copy that wrote them, no kernel ever writes there, and the image stays unmodified while the plan is used.  A table that a
// kernel fills would have to be read behind pdl_wait().
// Sender step of 64 tiles, back to back: 8.2 -> 6.3 us; no difference where the kernels are long.
// (early false: an ordinary launch.  For grids of a few blocks per SM that do not balance themselves: begun while a
// persistent kernel drains, they are packed onto the SMs that it leaves first.)
template <class... P, class... A>
cudaError_t launch_when(bool early, void (*kernel)(P...), dim3 grid, uint32_t threads, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, uint32_t threads, size_t smem, cudaStream_t s, A&&... args) {
    return launch_when(true, kernel, grid, threads, smem, s, args...);
}
// (and lets the kernel behind it begin in turn)
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
int check_launch();                            // cudaGetLastError -> status
void count_plan(int change);                   // plans that exist
// the persistent sender kernel with HashCache in place of the exponent cache (ciera_encode.cu)
int launch_encode_hashed(const ciera_plan* p, const void* weights_dev, void* hash_cache_dev, void* messages_dev,
                         uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, void* scratch, int32_t* status_dev,
                         cudaStream_t s);
// the argument checks of ciera_step; writes the outputs of units without values
int step_begin(const ciera_plan* p, const void* weights_dev, const void* sender_cache_dev, const void* msg_send_dev,
               const void* msg_recv_dev, const void* receiver_cache_dev, const void* weights_out_dev, uint64_t* wire_bytes_dev,
               uint32_t* changed_blocks_dev, const void* workspace_dev, cudaStream_t s);
// whether the buffers of a step lie apart, so that one launch may work on all of them
bool step_buffers_apart(const ciera_plan* p, const void* weights, const void* sender_cache, const void* msg_send,
                        const void* msg_recv, const void* receiver_cache, const void* weights_out);
// ciera_step on the tiles [lo, hi) of the plan's tiles by address; parts of one step go to one stream in order
int launch_step_part(const ciera_plan* p, const ciera_device_buffers* b, uint32_t lo, uint32_t hi, cudaStream_t s);
}  // namespace ciera
