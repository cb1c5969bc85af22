// Sender side (paper Algorithm 1, sender part; Section 3.1) as one persistent sm_100a kernel.
//
// Grid = G persistent thread blocks.  The plan lists the tiles of short units (up to 32 tiles)
// first.  A block first takes its share of the tiles of the longer units, spread tile by tile over
// the blocks (block c takes tiles T0 + c, T0 + c + G, ...; neighbouring tiles of a unit are then
// worked on by neighbouring blocks at about the same time, and their payload offsets come from a
// single-pass look-back over per-tile status words; with more than one tile to a block this part
// needs all blocks resident, so such a plan is launched cooperatively).  Then it works through the
// short units in runs of their tiles -- a long first run, a last run of at most four (see
// ciera_plan_create) --, drawing the next run's number from a counter in the scratch (every unit's
// first run goes out before any unit's second run, and so on): a tile's place in its unit's payload
// is then a running sum inside the block, which a run that does not start its unit takes over from
// the status word of the tile before it -- written many draws earlier -- and all SMs stay busy to the
// end whatever their individual pace (with whole units of 16 tiles as the piece of work drawn, the
// blocks finished up to a unit apart: 0.921 of the copy peak against 0.935).  Tables with few tiles in
// short units have all of their tiles spread (kSpreadShare).
// A thread block has four roles:
//
//   producer warp   runs ahead of the others: for each of its tiles it fetches the tile
//                   descriptor, works out the tile's addresses once for everybody, and starts two
//                   bulk-async copies into shared memory -- the weights tile into a short ring
//                   (freed as soon as the consumers have read it) and the cached-exponent tile
//                   into a longer ring (held until the tile's changed exponents have been sent);
//   16 consumer     each thread owns one or two pieces of consecutive values: split into exponent
//   warps           bytes and sign-plus-mantissa, compare with the cached exponents, vote (ballot)
//                   the "my piece changed" bit, store sign-plus-mantissa to the message and leave
//                   the new exponents where the cached ones were staged;
//   aggregator warp turns the vote bits of a tile into block flags (the unit's bitmap) and counts
//                   the tile's payload bytes; for a tile of a unit that this block works through
//                   alone it also keeps the running offset, otherwise it publishes the count as
//                   the tile's status word;
//   resolver warps  (spread tiles only) resolve the tile's exclusive offset in the unit's payload
//                   with a single-pass look-back over the status words.
// A few tiles later, when that offset is known, the consumers send the exponents of changed
// blocks from shared memory to the payload and to the cache and hand the stage back.
//
// Only the resolvers ever wait for another thread block; the aggregator never does, and the
// consumers only for a resolver that is several tiles late, so a tile's status is published as
// soon as its votes are in.
//
// The same kernel serves the sender that keeps HashCache (a 128-bit hash per block, Section 3.1 and
// Algorithm 1 as printed) instead of the previous exponents (template flag HASH): the producer then
// stages the tile's cached hashes instead of cached exponents, the consumers turn their exponents
// into hash terms and add them up over the lanes that share a block, and the aggregator finishes
// the hashes, compares them with the cached ones, refreshes HashCache and derives the block flags
// from the comparison.
//
// And it serves the whole step (template flag STEP, ciera_step): sender, transport and receiver of a table on one GPU.
// Bound by HBM, a step in three kernels writes each message, reads it, writes its copy and reads that: at q = 0.22
// 11.1 bytes per bf16 value move.  Here every byte of a message is stored to both buffers as it is made, and the
// consumers reconstruct a tile's weights from what travels (sign-plus-mantissa, exponents of changed blocks) and
// the receiver's cached exponents while the tile is still in shared memory: 8.9 bytes.  Measured per OLMoE-shaped
// layer, B = 512, q = 0.22: bf16 0.694 -> 0.572 ms (0.93 of the copy peak), fp32 1.436 -> 1.084 (0.94); every block
// changed, bf16: 0.933 -> 0.724.
//
// Whole steps on tables of long units have an instance of their own (template flag LONG, chosen by runs_as_long_units), which
// differs from the above in four things, explained where they stand: a block's spread tiles after the second are drawn from a
// counter (TileWalk); the look-back reads a short word per tile and a word per group of 32 tiles (look_back); both caches are
// refreshed as soon as a tile's flags are there, so that the exponents' ring is free once they are compared; and the payload
// goes out six tiles later, read back from the cache (EncodeLongCfg, FromCache).  A tile's votes, flags and offset then live
// in a ring of their own.
#include <cstddef>
#include <type_traits>

#include "ciera_bits.cuh"
#include "ciera_hash.cuh"
#include "ciera_lookback.cuh"
#include "ciera_pipe.cuh"

namespace ciera {

constexpr int kResolvers = 2;  // resolver warps (20 warps per block: two blocks per SM at 48 registers per thread)
// Consumer warps of a block, and how they share a tile.  With HashCache and 2-byte values, where the kernel is bound by
// instruction issue, 8 warps take four pieces a thread: what a warp spends on a tile as such (waits, addresses, sending)
// is spent half as often, and a warp's pieces are rows of 256 neighbouring values, so that rows of one block are added
// up in registers before anything is exchanged between lanes: OLMoE-shaped layer 0.357 -> 0.305 ms with 512 values per
// block (0.311 with inputs changing from pass to pass), 0.399 -> 0.361 with 64, 0.397 -> 0.319 with 4096.  (Three blocks per
// SM instead of two: 2 % faster with 512 values per block, 5 % slower with 64, small tables 8-15 % slower.  HASH == 3, whose
// consumers finish the hashes themselves, 0.494 -> 0.585: it keeps 16.)
template <int DT, int HASH>
constexpr int kConsumerWarps = (HASH == 1 || HASH == 2) && DT != CIERA_FP32 ? 8 : kWarps;
template <int DT, int HASH>
constexpr int kEncodeThreads = 32 * (kConsumerWarps<DT, HASH> + 2 + kResolvers);  // + producer, aggregator, resolvers
template <int DT, int CW>
struct Share {
    using P = Piece<DT>;
    static constexpr int kPerThread = kTileValues / (32 * CW * P::kValues);
    // first value (inside the tile) of piece p of consumer thread tid
    static __device__ __forceinline__ uint32_t start(uint32_t tid, int p) {
        if (CW == kWarps) return P::start(tid, p);
        return ((tid >> 5) * (uint32_t)kPerThread + (uint32_t)p) * (32u * P::kValues) + (tid & 31u) * P::kValues;
    }
};
constexpr uint32_t kRowL2 = 8;  // log2(values of a row) in the second layout
constexpr int kDescRing = 16;                                    // > exponent stages + 2
constexpr int kVoteWords = 32;  // vote bits of a tile: up to 1024 pieces

// Ring depths; kDefer = consumers send a tile's changed exponents this many tiles later.  With
// fine blocks (see ciera_internal.cuh) a tile has up to 8192 block flags instead of 512, and the
// exponent ring gives up a stage to make room for them (two thread blocks share an SM).
template <int DT, bool FINE>
struct EncodeCfg;
template <>
struct EncodeCfg<CIERA_BF16, false> {
    static constexpr int kWStages = 3;  // 3 x 16 KB weights tiles
    static constexpr int kEStages = 7;  // 7 x  8 KB exponent tiles
    static constexpr int kDefer = 3;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeCfg<CIERA_FP32, false> {
    static constexpr int kWStages = 2;  // 2 x 32 KB
    static constexpr int kEStages = 5;  // 5 x  8 KB
    static constexpr int kDefer = 3;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeCfg<CIERA_FP16, false> {  // as bf16: 16 KB weights tiles, 8 KB exponent tiles
    static constexpr int kWStages = 3;
    static constexpr int kEStages = 7;
    static constexpr int kDefer = 3;
    static constexpr int kBmWords = kBitmapWords;
};
// (fine blocks: the exponent ring is shorter still, to make room for the warps' gather spaces; ring depths of
// 3 + 5 with the sending two tiles later measured the same as 3 + 7 and three tiles later on the headline)
template <>
struct EncodeCfg<CIERA_BF16, true> {
    static constexpr int kWStages = 3;
    static constexpr int kEStages = 5;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kFineBitmapWords;
};
template <>
struct EncodeCfg<CIERA_FP16, true> : EncodeCfg<CIERA_BF16, true> {};  // the tile sizes of bf16
template <>
struct EncodeCfg<CIERA_FP32, true> {
    static constexpr int kWStages = 2;
    static constexpr int kEStages = 3;
    static constexpr int kDefer = 1;
    static constexpr int kBmWords = kFineBitmapWords;
};

// With HashCache the exponent ring stages no cached exponents (it only keeps the new ones until
// they are sent), so it is shorter; each of its stages has a companion with the tile's cached
// hashes and the consumers' partial sums, sized at launch from the block size.
// The template argument HASH of the kernel is 0 (exponent cache), 1 (HashCache), 2 (HashCache with
// shorter rings: with blocks of 64 values and fewer the hash stages are large, and two thread blocks
// still have to fit an SM) or 3 (as 2, and the consumers finish the blocks' hashes).
template <int DT, int HASH>
struct EncodeHashCfg;
template <>
struct EncodeHashCfg<CIERA_BF16, 1> {
    static constexpr int kWStages = 3;
    static constexpr int kEStages = 6;
    static constexpr int kDefer = 3;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeHashCfg<CIERA_FP32, 1> {
    static constexpr int kWStages = 2;
    static constexpr int kEStages = 4;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeHashCfg<CIERA_FP16, 1> : EncodeHashCfg<CIERA_BF16, 1> {};  // fp16: the tile sizes of bf16
template <>
struct EncodeHashCfg<CIERA_BF16, 2> {
    static constexpr int kWStages = 3;
    static constexpr int kEStages = 4;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeHashCfg<CIERA_FP32, 2> {
    static constexpr int kWStages = 2;
    static constexpr int kEStages = 3;
    static constexpr int kDefer = 1;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeHashCfg<CIERA_FP16, 2> : EncodeHashCfg<CIERA_BF16, 2> {};
template <int DT>
struct EncodeHashCfg<DT, 3> : EncodeHashCfg<DT, 2> {};
constexpr uint32_t kHashShortRingsLog2 = 6;  // blocks of up to 2^6 values take the shorter rings
// With 256 and more blocks in a tile (16 and 32 values per block) the consumers finish the blocks' hashes
// themselves: kernel instance HASH == 3 (see finish_hash_groups; blocks of at least two lanes' pieces).
constexpr uint32_t kHashByConsumersLog2 = 5;
// The whole-step kernel (STEP) also stages the receiver's cached exponents, behind each weights tile.  With coarse
// blocks the weights stage is held until the tile's block flags are there, one slot later, so that a third stage
// counts: bf16 with 3 + 4 stages 0.571 ms per OLMoE-shaped layer, with 2 + 6 0.628.  fp32 has room for it only with one
// thread block per SM: 1.080 ms with 4 + 5 stages, 1.459 with two blocks of 2 + 3.  (Reconstructing at once from
// the votes of the own warp, for blocks that lie in one warp's pieces: bf16 0.582, fp32 1.084 ms.)
template <int DT, bool FINE>
struct EncodeStepCfg;
template <>
struct EncodeStepCfg<CIERA_BF16, false> {
    static constexpr int kWStages = 3;  // 3 x (16 + 8) KB
    static constexpr int kEStages = 4;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeStepCfg<CIERA_FP32, false> {
    static constexpr int kWStages = 4;  // 4 x (32 + 8) KB
    static constexpr int kEStages = 5;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kBitmapWords;
};
template <>
struct EncodeStepCfg<CIERA_FP16, false> : EncodeStepCfg<CIERA_BF16, false> {};
template <>
struct EncodeStepCfg<CIERA_BF16, true> {
    static constexpr int kWStages = 2;
    static constexpr int kEStages = 5;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kFineBitmapWords;
};
template <>
struct EncodeStepCfg<CIERA_FP16, true> : EncodeStepCfg<CIERA_BF16, true> {};
template <>
struct EncodeStepCfg<CIERA_FP32, true> {
    static constexpr int kWStages = 3;
    static constexpr int kEStages = 5;
    static constexpr int kDefer = 2;
    static constexpr int kBmWords = kFineBitmapWords;
};
// LONG, the whole step on tables of long units (coarse blocks).  What bounds these tables is not memory but that every tile waits
// for the votes of all tiles before it in its unit: loads take 3 to 12 us when hundreds of tiles are in flight, and blocks
// that were two tiles from their oldest unsent payload stood still for the slowest (one tensor of 2^28 bf16 values on 4 shards:
// 477 us, with made-up offsets 414, and 370 if in addition blocks may take tiles at their own pace).  So the exponents' ring only
// holds the cached ones until they are compared, both caches are refreshed as soon as a tile's flags are there, its payload goes
// out kDefer tiles later from the cache (see FromCache), tiles are drawn (see TileWalk), and the look-back reads groups: 394 us,
// 0.90 of the copy peak.  Of these drawing is worth the least and not always something: given out by block number 395 us, one
// tensor of 2^26 bf16 values 116 (drawn 112), 2^27 fp32 398 (392), 2^26 fp16 139 (132), 2^28 fp16 472 (483).  In runs of short
// units, where offsets need no look-back, the other instance is as fast or faster (see runs_as_long_units).
template <int DT>
struct EncodeLongCfg {
    static constexpr int kWStages = DT == CIERA_FP32 ? 4 : 3;
    static constexpr int kEStages = DT == CIERA_FP32 ? 4 : 3;
    static constexpr int kDefer = 6;
    static constexpr int kBmWords = kBitmapWords;
};
template <int DT, bool STEP>
constexpr int kEncodeBlocksPerSM = STEP && DT == CIERA_FP32 ? 1 : 2;
// Values of changed blocks from which a tile counts as dense, rounded down to whole blocks: three of four with 2048 values per
// block and one of two with 4096, where pieces that are missing lie in long stretches.  (Half an OLMoE-shaped layer, 0.57 of
// the blocks of 4096 changed: bf16 331 us, 338 with two of two; fp32 581 and 590; 2048, 0.59 changed, 338 and 342.)
constexpr uint32_t kDenseValues = (uint32_t)kTileValues / 8u * 7u;
template <int DT, bool FINE, int HASH, bool STEP, bool LONG = false>
struct EncodeCfgOf {
    using type = EncodeHashCfg<DT, HASH>;
};
template <int DT, bool FINE>
struct EncodeCfgOf<DT, FINE, 0, false> {
    using type = EncodeCfg<DT, FINE>;
};
template <int DT, bool FINE>
struct EncodeCfgOf<DT, FINE, 0, true> {
    using type = EncodeStepCfg<DT, FINE>;
};
template <int DT>
struct EncodeCfgOf<DT, false, 0, true, true> {
    using type = EncodeLongCfg<DT>;
};
// A tile's votes, flags and offset live in a ring of their own; it is as long as the ring of exponents, which waits for the
// sending too, but for LONG.
template <class Cfg, bool LONG>
constexpr int kResultStages = LONG ? Cfg::kDefer + 1 : Cfg::kEStages;

// Distances, in bytes, from the sender's buffers to their counterparts on the receiver's side (STEP; else unused):
// unit layouts are the same on both sides, so one distance serves a whole buffer.
struct StepTwins {
    int64_t msg;      // sent messages -> received messages
    int64_t cache;    // sender's exponent cache -> receiver's
    int64_t weights;  // weights -> reconstructed weights
};

// Shared-memory bytes of the cached hashes (`hold`) and of the partial sums (`part`) of one tile:
// 16 bytes per block, and 16 bytes per group of lanes that add up their terms (a block's lanes, at
// most a warp).
template <int DT>
__host__ __device__ constexpr uint32_t hash_hold_bytes(uint32_t log2b) {
    return (uint32_t)(kTileValues >> log2b) * 16u;
}
template <int DT>
__host__ __device__ constexpr uint32_t hash_part_bytes(uint32_t log2b) {
    const uint32_t nbt = (uint32_t)kTileValues >> log2b;
    const uint32_t warps = (uint32_t)kTileValues >> (5 + Piece<DT>::kLog2Values);  // warp-sized groups of pieces
    return (nbt > warps ? nbt : warps) * 16u;
}

// What the consumers need of a tile, worked out once by the producer thread instead of by each
// of the 512 consumer threads.
struct __align__(16) EncodeTileInfo {
    uint8_t* sm_dst;       // where the tile's sign-plus-mantissa goes
    uint8_t* pay_dst;      // start of the unit's payload section
    uint8_t* c_ptr;        // the tile's cached exponents (with HashCache: the cached hash of the tile's first block)
    const uint8_t* w_src;  // the tile's weights
    uint32_t nv;           // values in the tile
    uint32_t r_staged;     // STEP: the receiver's cached exponents are staged (else the few needed are read where they lie)
    uint32_t pad[2];
};

// The tiles whose last 16-byte piece reaches behind the last value of the weights buffer or of an exponent cache
// (kNoTile: there is none); several: there are more, and every short tile is taken for one.
struct BufferEnds {
    uint32_t weights, cache;
    bool several;
    __device__ __forceinline__ bool has(uint32_t tile, uint32_t nv) const {
        return tile == weights || tile == cache || (several && (nv & 15u));
    }
};

// Producer, a tile that ends a buffer: bulk copies as far as whole 16-byte pieces go, small copies that stop in time for
// the rest, all on `bar`.  (st_e null: no cached exponents; r_at: where behind the staged weights the receiver's go, 0 =
// nowhere, and r_twin their distance.  Not inlined: at 48 registers per thread the producer's loop spills more for what it
// might need here.  Steps of 12 288 units of 4 688 values 117 us inlined, 115 like this, 118 with the consumers fetching
// the broken pieces, 113 when all that lies in the last 16 bytes was read, whether there or not.)
__device__ __noinline__ void stage_buffer_end(uint8_t* st_w, const uint8_t* w, uint32_t w_bytes, uint8_t* st_e, const uint8_t* e,
                                              uint32_t e_bytes, uint32_t r_at, int64_t r_twin, uint64_t* bar) {
    const uint32_t w_whole = w_bytes & ~15u, e_whole = st_e ? e_bytes & ~15u : 0u;
    mbar_expect_tx(bar, w_whole + e_whole + (r_at ? e_whole : 0u));
    if (w_whole) bulk_load(st_w, w, w_whole, bar);
    if (w_bytes & 15u) cp_async16_first(st_w + w_whole, w + w_whole, w_bytes & 15u);
    if (e_whole) {
        bulk_load(st_e, e, e_whole, bar);
        if (r_at) bulk_load(st_w + r_at, e + r_twin, e_whole, bar);
    }
    if (st_e && (e_bytes & 15u)) {
        cp_async16_first(st_e + e_whole, e + e_whole, e_bytes & 15u);
        if (r_at) cp_async16_first(st_w + r_at + e_whole, e + r_twin + e_whole, e_bytes & 15u);
    }
    cp_async_arrive(bar);
    mbar_arrive(bar);
}

template <int SW, int SE, int SR, int BW>
struct EncodeCtl {
    uint64_t full_w[SW];    // weights tile landed
    uint64_t empty_w[SW];   // all 16 consumer warps have read it
    uint64_t full_e[SE];    // cached-exponent tile landed
    uint64_t voted[SR];     // all 16 consumer warps have left their exponents there and voted
    uint64_t summed[SR];    // aggregator has published the tile's status and block flags
    uint64_t resolved[SR];  // a resolver knows the tile's offset in the unit's payload
    uint64_t empty_e[SE];   // all 16 consumer warps have sent the tile's changed exponents
    TileDesc desc[kDescRing];
    EncodeTileInfo info[kDescRing];
    uint32_t tile_idx[kDescRing];  // table index of the tile in desc[]; kNoTile = end marker
    uint32_t seq[kDescRing];       // kSeq* bits: tile of a run that this block works through alone, first / last of the run
    uint32_t ballot[SR][kVoteWords];  // coarse blocks: "my piece differs" votes
    uint32_t bm[SR][BW];              // block flags of the tile (16-byte aligned: checked where the kernel starts)
    uint16_t pre[SR][BW];             // set flags before each word of bm
    unsigned long long agg[SR];
    unsigned long long base[SR];
    int abort;
    uint32_t issued;  // tiles whose loads have been started (producer)
    uint32_t seen;    // tiles whose loads the consumers have seen complete
};

constexpr uint32_t kEarlyClearTiles = 4096;  // status words that one warp empties while the rest still works

// How a tile relates to the run of tiles it was handed out with (a short unit's tiles go out in runs of
// kSeqRunTiles, see ciera_internal.cuh): bit 0 = the tile belongs to a run (else: a spread tile of a longer
// unit), bit 1 = first tile of its run, bit 2 = last tile of its run.
constexpr uint32_t kSeqTile = 1u, kSeqRunStart = 2u, kSeqRunEnd = 4u;

// The sequence of tiles of one thread block (see the head of this file); used by the producer.
// Runs of the short units: block b starts with runs b and b + G (no round trip to the counter stands between
// the start of the kernel and the first loads); every run taken is paid for with one draw from the counter, so
// the counter is drawn from exactly n_runs times in a launch, and the thread that makes the last draw puts it
// back to zero for the next launch.  The walk keeps two runs in hand besides the current one: the number of
// the run after next (its draw is on its way) and the table entry of the next run (its load is on its way), so
// that at the start of a run neither the counter nor the table is waited for.
// DRAWN (LONG): a block's spread tiles after the second are drawn from a counter of their own, from exactly n_spread - G times,
// so that blocks may work at their own pace.  All later tiles of a tile's unit wait for its votes, so it must not be held long:
// the number of tile k + 2 is drawn, and the descriptor of tile k + 1 fetched, when the loads of tile k have been started.
// Later is worse, since the round trips to counter and descriptor then stand in the producer's way (one tensor of 2^28 bf16
// values on 4 shards 397 us; tile k + 1 drawn and fetched when the loads of tile k have been started 405, when its stage is
// free 435; 2^27 fp32 values 392, 396, 417).
template <bool ORDERED, bool DRAWN>  // ORDERED: the spread tiles may be given by their places in a list (steps in parts)
struct TileWalk {
    const uint2* seq_runs;
    const uint32_t* order;  // not null: the spread tiles are given by their places in this list
    unsigned int* run_ticket;
    uint32_t n_tiles, n_runs, G;
    uint32_t tile, end;      // current run: next tile, one past its last tile
    uint2 next_range;        // the next run's tiles (valid if next_run < n_runs)
    uint32_t next_run;       // number of the next run
    uint32_t after_run;      // number of the run after that
    uint32_t spread_tile;    // next spread tile of this block, or its number as drawn
    uint32_t first_drawn;    // DRAWN: the tile with drawn number 0
    uint32_t taken;          // DRAWN: spread tiles so far
    bool spread;

    __device__ TileWalk(const uint2* runs, const uint32_t* places, unsigned int* ticket, uint32_t nruns, uint32_t spread_first, uint32_t nt,
                        uint32_t grid, uint32_t block)
        : seq_runs(runs), order(places), run_ticket(ticket), n_tiles(nt), n_runs(nruns), G(grid), tile(0), end(0),
          first_drawn(spread_first + 2u * grid), taken(0), spread(true) {
        spread_tile = spread_first + block;  // tiles of longer units start after the short units' tiles
        next_run = block;
        after_run = block + grid;
        next_range = make_uint2(0u, 0u);
        if (next_run < n_runs) next_range = __ldg(seq_runs + next_run);
    }
    __device__ uint32_t draw() {
        const uint32_t d = atomicAdd(run_ticket, 1u);
        if (d + 1u == n_runs) atomicExch(run_ticket, 0u);  // that was the launch's last draw
        return d + 2u * G;
    }
    // next tile, or kNoTile; `seq` gets the kSeq* bits of the tile
    __device__ uint32_t next(uint32_t& seq) {
        if (spread) {
            uint32_t at = spread_tile;
            if (DRAWN && taken >= 2u) {
                at += first_drawn;
                if (at + 1u == n_tiles + G) atomicExch(run_ticket + 2, 0u);  // that was the launch's last draw
            }
            if (at < n_tiles) {
                seq = 0;
                const uint32_t t = ORDERED && order ? __ldg(order + at) : at;
                spread_tile = !DRAWN || taken == 0u ? at + G : atomicAdd(run_ticket + 2, 1u);
                if (DRAWN) ++taken;
                return t;
            }
            spread = false;
        }
        seq = kSeqTile;
        while (tile == end) {
            if (next_run >= n_runs) return kNoTile;
            tile = next_range.x;
            end = next_range.y;
            next_run = after_run;
            if (next_run < n_runs) next_range = __ldg(seq_runs + next_run);
            after_run = draw();
            seq |= kSeqRunStart;
        }
        if (tile + 1u == end) seq |= kSeqRunEnd;
        return tile++;
    }
    // the next call of next() returns a drawn tile: it is fetched, and the one after it drawn, when this tile's loads have been started
    __device__ bool late() const { return DRAWN && spread && taken >= 2u; }
};

// The first tile that the walk of `block` will hand out, from the tables alone.
template <bool ORDERED>
__device__ __forceinline__ uint32_t first_tile(const uint2* runs, const uint32_t* places, uint32_t n_runs, uint32_t spread_first,
                                               uint32_t n_tiles, uint32_t block) {
    const uint32_t at = spread_first + block;
    if (at < n_tiles) return ORDERED && places ? __ldg(places + at) : at;
    return block < n_runs ? __ldg(runs + block).x : kNoTile;
}

// Fine blocks: the consumers have written the block flags themselves; fills pre (set bits before
// each word) and returns the number of changed blocks of the tile (one warp).
// Lane l takes the W = nwords / 32 consecutive words l W .. l W + W - 1 (1, 2, 4 or 8), so that one scan over
// the lanes does for the whole tile.
template <int W>
__device__ __forceinline__ uint32_t scan_block_bitmap_w(const uint32_t* bm, uint16_t* pre, uint32_t lane) {
    uint32_t w[W];
    if constexpr (W >= 4) {
#pragma unroll
        for (int i = 0; i < W / 4; ++i) {
            const uint4 v = reinterpret_cast<const uint4*>(bm)[lane * (W / 4) + i];
            w[4 * i] = v.x; w[4 * i + 1] = v.y; w[4 * i + 2] = v.z; w[4 * i + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < W; ++i) w[i] = bm[lane * W + i];
    }
    uint32_t before[W], sum = 0;
#pragma unroll
    for (int i = 0; i < W; ++i) {
        before[i] = sum;
        sum += __popc(w[i]);
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += t;
    }
    const uint32_t base = incl - sum;
    if constexpr (W >= 2) {  // two 16-bit counts per store
        uint32_t* pre32 = reinterpret_cast<uint32_t*>(pre) + lane * (W / 2);
#pragma unroll
        for (int i = 0; i < W / 2; ++i) pre32[i] = (base + before[2 * i]) | ((base + before[2 * i + 1]) << 16);
    } else {
        pre[lane] = (uint16_t)base;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    __syncwarp();
    return total;
}
__device__ __forceinline__ uint32_t scan_block_bitmap(const uint32_t* bm, uint16_t* pre, uint32_t log2b, uint32_t lane) {
    if (log2b == 0) return scan_block_bitmap_w<8>(bm, pre, lane);  // 256 words: eight per lane, one scan
    if (log2b == 1) return scan_block_bitmap_w<4>(bm, pre, lane);  // 128 words: four per lane
    const uint32_t nwords = kTileValues >> (log2b + 5);  // 32 .. 128: a scan per 32 words
    uint32_t run = 0;
    for (uint32_t base = 0; base < nwords; base += 32) {
        const uint32_t pc = __popc(bm[base + lane]);
        uint32_t incl = pc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += t;
        }
        pre[base + lane] = (uint16_t)(run + incl - pc);
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    return run;
}

// Blocks whose hashes the consumers finish themselves (see finish_hash_groups; kernel instance HASH == 3): many
// per tile, and made of at least two lanes' pieces.
template <int DT>
__host__ __device__ __forceinline__ bool hash_finished_by_consumers(uint32_t log2b) {
    return log2b <= kHashByConsumersLog2 && log2b > (uint32_t)Piece<DT>::kLog2Values;
}

// Aggregator warp, one tile: block flags, the tile's bitmap bytes, the tile's payload byte count.
// With `publish` the count goes out at once as the tile's status word, so that later tiles never
// wait for it longer than for the votes themselves.  Waits for nothing outside the thread block.
// HashCache: block flags of a tile from the consumers' partial sums.  Lane i of a round takes one
// block: adds up the block's partial sums, finishes the two hashes, compares them with the cached
// pair and, where they differ, flags the block and stores the new pair (HashCache[i,k] <- h).
// Returns the number of flagged blocks (one warp).
template <int DT, bool BY_CONSUMERS>
__device__ __forceinline__ uint32_t hash_block_bitmap(const ulonglong2* part, const ulonglong2* hold, ulonglong2* hash_dst,
                                                      uint32_t* bm, uint16_t* pre, uint32_t log2b, uint32_t nv,
                                                      uint32_t lane) {
    // log2(values behind a partial sum): a warp's pieces, or in rows (8 consumer warps) all four of its rows
    constexpr uint32_t kGroupL2 = kConsumerWarps<DT, 1> == kWarps ? 5 + Piece<DT>::kLog2Values : kRowL2 + 2;
    const uint32_t B = 1u << log2b;
    const uint32_t nbt = kTileValues >> log2b;
    const uint32_t nblk = (nv + B - 1u) >> log2b;
    const uint32_t epb_l2 = log2b > kGroupL2 ? log2b - kGroupL2 : 0u;  // log2(partial sums per block)
    const uint8_t* const verdicts = reinterpret_cast<const uint8_t*>(part);
    // one block: true iff its hashes differ from the cached pair (which is then replaced)
    auto finish_block = [&](uint32_t i) -> bool {
        if (i >= nblk) return false;
        if (BY_CONSUMERS) return verdicts[i] != 0;  // finished, compared and stored by the consumers already
        uint64_t a = 0, b = 0;
        for (uint32_t e = 0; e < (1u << epb_l2); ++e) {
            const ulonglong2 v = part[(i << epb_l2) + e];
            a += v.x;
            b += v.y;
        }
        const ulonglong2 h = hash_finish(a, b, min(B, nv - (i << log2b)));
        const ulonglong2 old = hold[i];
        const bool f = h.x != old.x || h.y != old.y;
        if (f) hash_dst[i] = h;
        return f;
    };
    uint32_t run = 0;
    uint32_t base = 0;
    // two blocks per lane and round while there are 64 and more (their chains of multiplies overlap; four were slower)
    for (; base + 64 <= nbt; base += 64) {
        const bool f0 = finish_block(base + lane), f1 = finish_block(base + 32 + lane);
        const uint32_t w0 = __ballot_sync(0xffffffffu, f0), w1 = __ballot_sync(0xffffffffu, f1);
        if (lane == 0) {
            bm[base >> 5] = w0;
            pre[base >> 5] = (uint16_t)run;
            bm[(base >> 5) + 1] = w1;
            pre[(base >> 5) + 1] = (uint16_t)(run + __popc(w0));
        }
        run += __popc(w0) + __popc(w1);
    }
    for (; base < nbt; base += 32) {
        const uint32_t word = __ballot_sync(0xffffffffu, finish_block(base + lane));
        if (lane == 0) {
            bm[base >> 5] = word;
            pre[base >> 5] = (uint16_t)run;
        }
        run += __popc(word);
    }
    __syncwarp();
    return run;
}

// HashCache, consumers: adds up the pieces' sums of terms (a[p], b[p]: the two hashes' sums of piece
// p of this thread) over groups of 2^l2 neighbouring lanes -- the lanes whose pieces lie in one block,
// at most the warp -- and stores the group's totals as entry e0 (piece 0) and e1 (the thread's last
// piece) of `part`, two 64-bit words each.  Instead of one butterfly per sum, the first exchanges
// hand every lane fewer sums to carry on with (odd lanes keep the b's, even lanes the a's; then lanes
// with bit 1 set keep the second piece's): 6 shuffles of 64 bits for four sums over a warp, not 20.
template <int NP>
__device__ __forceinline__ void reduce_hash_terms(const uint64_t* a, const uint64_t* b, uint32_t l2, uint32_t e0, uint32_t e1,
                                                  uint64_t* part, uint32_t lane) {
    const bool odd = (lane & 1u) != 0;
    if (l2 == 0) {  // every lane a block of its own (NP = 1: a piece is a whole block at least)
        part[2 * e0] = a[0];
        part[2 * e0 + 1] = b[0];
        return;
    }
    uint64_t k0 = (odd ? b[0] : a[0]) + __shfl_xor_sync(0xffffffffu, odd ? a[0] : b[0], 1);
    if constexpr (NP == 1) {
#pragma unroll
        for (uint32_t o = 1; o < 5; ++o)
            if (o < l2) k0 += __shfl_xor_sync(0xffffffffu, k0, 1u << o);
        const uint32_t r = lane & ((1u << l2) - 1u);
        if (r < 2) part[2 * e0 + r] = k0;  // lane 0 of the group: sum of a, lane 1: sum of b
    } else {
        uint64_t k1 = (odd ? b[1] : a[1]) + __shfl_xor_sync(0xffffffffu, odd ? a[1] : b[1], 1);
        if (l2 == 1) {  // groups of two lanes
            part[2 * e0 + (odd ? 1u : 0u)] = k0;
            part[2 * e1 + (odd ? 1u : 0u)] = k1;
            return;
        }
        const bool second = (lane & 2u) != 0;
        uint64_t t = (second ? k1 : k0) + __shfl_xor_sync(0xffffffffu, second ? k0 : k1, 2);
#pragma unroll
        for (uint32_t o = 2; o < 5; ++o)
            if (o < l2) t += __shfl_xor_sync(0xffffffffu, t, 1u << o);
        const uint32_t r = lane & ((1u << l2) - 1u);
        if (r < 4) part[2 * ((r & 2u) ? e1 : e0) + (r & 1u)] = t;  // lanes 0..3: a of piece 0, b of piece 0, a, b of piece 1
    }
}

// The same for four rows of one warp (see Share): rows that lie in one block are added up first, entry of a group =
// index of its values in units of the smaller of block and warp.  v0: the first value of this thread.  Blocks of 64 values and more (l2 >= 3); 9, 6 or 5 shuffles
// of 64 bits for blocks of up to 256, 512, or 1024 values and more.
__device__ __forceinline__ void reduce_hash_rows(uint64_t (&a)[4], uint64_t (&b)[4], uint32_t l2, uint32_t log2b, uint32_t v0,
                                                 uint64_t* part, uint32_t lane) {
    if (log2b > kRowL2 + 1) {
        const uint64_t sa = (a[0] + a[1]) + (a[2] + a[3]), sb = (b[0] + b[1]) + (b[2] + b[3]);
        reduce_hash_terms<1>(&sa, &sb, 5u, v0 >> (kRowL2 + 2), 0u, part, lane);
        return;
    }
    if (log2b == kRowL2 + 1) {
        const uint64_t sa[2] = {a[0] + a[1], a[2] + a[3]}, sb[2] = {b[0] + b[1], b[2] + b[3]};
        reduce_hash_terms<2>(sa, sb, 5u, v0 >> log2b, (v0 >> log2b) + 1u, part, lane);
        return;
    }
    const bool odd = (lane & 1u) != 0, second = (lane & 2u) != 0, third = (lane & 4u) != 0;
    uint64_t k[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) k[p] = (odd ? b[p] : a[p]) + __shfl_xor_sync(0xffffffffu, odd ? a[p] : b[p], 1);
    const uint64_t t0 = (second ? k[1] : k[0]) + __shfl_xor_sync(0xffffffffu, second ? k[0] : k[1], 2);
    const uint64_t t1 = (second ? k[3] : k[2]) + __shfl_xor_sync(0xffffffffu, second ? k[2] : k[3], 2);
    uint64_t u = (third ? t1 : t0) + __shfl_xor_sync(0xffffffffu, third ? t0 : t1, 4);
#pragma unroll
    for (uint32_t o = 3; o < 5; ++o)
        if (o < l2) u += __shfl_xor_sync(0xffffffffu, u, 1u << o);
    // lanes 0..7 of a group: bit 0 which sum, bits 1 and 2 the row
    const uint32_t r = lane & ((1u << l2) - 1u);
    if (r < 8u) part[2u * ((v0 + ((r >> 1) << kRowL2)) >> log2b) + (r & 1u)] = u;
}

// HashCache, consumers, kernel instance HASH == 3 (blocks that lie inside one warp's pieces and span at least two
// lanes, l2 >= 1): the same reduction as reduce_hash_terms, but the lanes that end up with a block's sums
// finish the block themselves -- each finishes one 64-bit half, compares it with its cached half, and the two
// halves of a block (in neighbouring lanes) agree on the verdict with one exchange; a changed block's new hash
// goes to HashCache at once (HashCache[i,k] <- h), and one byte per block tells the aggregator the verdict.
// With 256 or 512 blocks in a tile the one aggregator warp, finishing them all by itself, set the pace of the
// whole thread block (0.82 ms per layer with 32 values per block, 1.24 ms with 16, whatever the change rate);
// with fewer blocks per tile the extra work in the consumers costs more than it saves (measured), so those
// keep the aggregator's way.
//   hold   the tile's cached hashes (two words per block), staged in shared memory
//   dst    the same in global memory
//   flags  one byte per block of the tile (written for every block below nblk)
template <int DT, int NP>
__device__ __forceinline__ void finish_hash_groups(const uint64_t* a, const uint64_t* b, uint32_t l2, uint32_t log2b,
                                                   uint32_t nv, uint32_t tid, const uint64_t* hold, uint64_t* dst,
                                                   uint8_t* flags, uint32_t lane) {
    using P = Piece<DT>;
    const bool odd = (lane & 1u) != 0;
    const uint32_t B = 1u << log2b;
    // One half of one block: `t` = the sum of the half's terms over the block (held by `leader` lanes, the half is
    // the lane's parity), `piece` = which of the thread's pieces lies in that block.  Called by all lanes together.
    auto finish_half = [&](uint64_t t, int piece, bool leader) {
        const uint32_t blk = P::start(tid, piece) >> log2b;
        const uint32_t first = blk << log2b;
        const bool mine = leader && first < nv;
        uint64_t h = 0;
        uint32_t differs = 0;
        if (mine) {
            h = mix64(t + min(B, nv - first));
            differs = h != hold[2u * blk + (odd ? 1u : 0u)] ? 1u : 0u;
        }
        differs |= __shfl_xor_sync(0xffffffffu, differs, 1);  // the block's two halves sit in neighbouring lanes
        if (mine) {
            if (differs) dst[2u * blk + (odd ? 1u : 0u)] = h;
            if (!odd) flags[blk] = (uint8_t)differs;
        }
    };
    const uint32_t r = lane & ((1u << l2) - 1u);
    uint64_t k0 = (odd ? b[0] : a[0]) + __shfl_xor_sync(0xffffffffu, odd ? a[0] : b[0], 1);
    if constexpr (NP == 1) {
#pragma unroll
        for (uint32_t o = 1; o < 5; ++o)
            if (o < l2) k0 += __shfl_xor_sync(0xffffffffu, k0, 1u << o);
        finish_half(k0, 0, r < 2u);
    } else {
        const uint64_t k1 = (odd ? b[1] : a[1]) + __shfl_xor_sync(0xffffffffu, odd ? a[1] : b[1], 1);
        if (l2 == 1) {  // a block is two lanes' pieces: every lane finishes a half of each of its two blocks
            finish_half(k0, 0, true);
            finish_half(k1, NP - 1, true);
        } else {
            const bool second = (lane & 2u) != 0;
            uint64_t t = (second ? k1 : k0) + __shfl_xor_sync(0xffffffffu, second ? k0 : k1, 2);
#pragma unroll
            for (uint32_t o = 2; o < 5; ++o)
                if (o < l2) t += __shfl_xor_sync(0xffffffffu, t, 1u << o);
            finish_half(t, second ? NP - 1 : 0, r < 4u);
        }
    }
}

// what aggregate_tile needs besides the votes when the sender keeps HashCache
struct HashTile {
    const ulonglong2* part;
    const ulonglong2* hold;
    ulonglong2* dst;
};

template <int DT, bool FINE, int HASH, class WORD>
__device__ __forceinline__ uint64_t aggregate_tile(const TileDesc& td, uint32_t tile, uint32_t log2b, bool publish,
                                                   const uint32_t* ballot, uint32_t* bm, uint16_t* pre,
                                                   WORD* tile_status, unsigned long long* groups, const HashTile& ht, uint32_t nv,
                                                   uint32_t lane) {
    const uint32_t B = 1u << log2b;
    const uint32_t nbt = kTileValues >> log2b;

    uint32_t run;
    if constexpr (HASH)
        run = hash_block_bitmap<DT, HASH == 3>(ht.part, ht.hold, ht.dst, bm, pre, log2b, nv, lane);
    else
        run = FINE ? scan_block_bitmap(bm, pre, log2b, lane)
                   : build_block_bitmap(ballot, bm, pre, log2b, Piece<DT>::kLog2Values, lane);

    // payload bytes of this tile: B per changed block, less for a changed short last block
    uint64_t agg = payload_bytes_of_blocks<DT>(run, log2b);
    const uint32_t rem = nv & (B - 1u);
    if (rem) {
        const uint32_t kb = nv >> log2b;
        if ((bm[kb >> 5] >> (kb & 31u)) & 1u) agg -= block_payload_bytes(B, DT) - block_payload_bytes(rem, DT);
    }
    if (publish) {
        const uint32_t mybits = nbt < 8 ? bm[0] : 0u;
        if constexpr (sizeof(WORD) == 4) {
            if (lane == 0) report_tile(tile_status, groups, td, tile, mybits, (uint32_t)agg);
        } else {
            // a unit's first tile knows its prefix (0) already
            const unsigned long long flag = td.tile_in_unit == 0 ? kFlagPrefix : kFlagAggregate;
            if (lane == 0) st_status(tile_status + tile, flag | ((unsigned long long)mybits << kBitsShift) | agg);
        }
    }
    return agg;
}

// The tile's bytes of the bitmap (tiles of >= 8 blocks own whole bytes).  `dst`: where they go; `nblk`: blocks of the tile.
// Fine blocks: at least 128 bytes per full tile, starting on a 128-byte boundary of the (16-byte aligned) slot.
template <bool STEP>
__device__ __forceinline__ void store_bitmap_fine(uint8_t* dst, const uint32_t* bm, uint32_t nblk, const StepTwins& tw,
                                                  uint32_t lane) {
    const uint32_t nbytes = (nblk + 7u) >> 3;
    uint32_t* const dst32 = reinterpret_cast<uint32_t*>(dst);
    uint32_t* const twin32 = reinterpret_cast<uint32_t*>(dst + tw.msg);
    // 16 bytes at a time, then the last words, then the last bytes
    const uint32_t quads = nbytes >> 4;
    for (uint32_t c = lane; c < quads; c += 32) {
        const uint4 v = reinterpret_cast<const uint4*>(bm)[c];
        reinterpret_cast<uint4*>(dst32)[c] = v;
        if (STEP) reinterpret_cast<uint4*>(twin32)[c] = v;
    }
    for (uint32_t w = 4u * quads + lane; w < (nbytes >> 2); w += 32) {
        dst32[w] = bm[w];
        if (STEP) twin32[w] = bm[w];
    }
    const uint32_t done = nbytes & ~3u;
    if (lane < nbytes - done) put_byte<STEP>(dst + done + lane, (uint8_t)(bm[done >> 2] >> (lane * 8u)), tw.msg);
}
// Coarse blocks: lane l holds word l of the flags; a tile of 32 blocks and more starts on a word boundary.
template <bool STEP>
__device__ __forceinline__ void store_bitmap(uint8_t* dst, uint32_t word, uint32_t nblk, const StepTwins& tw, uint32_t lane) {
    const uint32_t nbytes = (nblk + 7u) >> 3;
    if (4u * lane + 4u <= nbytes) {
        *reinterpret_cast<uint32_t*>(dst + 4u * lane) = word;
        if (STEP) *reinterpret_cast<uint32_t*>(dst + tw.msg + 4u * lane) = word;
    } else {
        for (uint32_t b = 4u * lane; b < nbytes; ++b) put_byte<STEP>(dst + b, (uint8_t)(word >> ((b & 3u) * 8u)), tw.msg);
    }
}

// payload <- exponents of changed blocks in block order; cache refreshed for the same blocks.
// Every consumer thread sends the exponents of its own pieces if their block changed; `source(x, p, t0, nvalid)` puts those of
// piece p into x, and `base` is the tile's exclusive offset in the unit's payload.
// (CACHE = false, the sender with HashCache, and LONG: payload only.)
// (FULL: the tile is a full one, every piece complete.)
// (STEP: the same bytes also go to the received message and to the receiver's cache.)
template <int DT, bool CACHE, bool FULL, bool STEP, class SHARE, class SOURCE>
__device__ __forceinline__ void write_changed(const EncodeTileInfo& ti, uint32_t log2b, const uint32_t* bm,
                                              const uint16_t* pre, uint64_t base, const StepTwins& tw, uint32_t tid, SOURCE source) {
    using P = Piece<DT>;
#pragma unroll
    for (int p = 0; p < SHARE::kPerThread; ++p) {
        const uint32_t t0 = SHARE::start(tid, p);
        const int nvalid = FULL ? (int)P::kValues : piece_valid<DT>(t0, ti.nv);
        if (nvalid == 0) continue;
        const uint32_t kb = t0 >> log2b;
        const uint32_t word = bm[kb >> 5];
        const bool changed = (word >> (kb & 31u)) & 1u;
        if constexpr (DT == CIERA_FP16 && FULL && STEP) {
            // Blocks of 32 values and more: four neighbouring lanes' pieces make 20 bytes = 5 aligned words.  Lane a
            // of the four writes word a -- the top of its neighbour's 40 bits, then its own -- and lane 3 the last one.
            // Ten byte stores per piece and message pair bound the step by issue and LSU: with the words, the gathered
            // sign-plus-mantissa and the exchange of exponents in place an OLMoE-shaped fp16 layer takes 0.600 ms
            // instead of 0.677 at 32 values per block, 0.611 instead of 0.652 at 512 (its bytes: 0.57 ms at the copy
            // peak).  The sender alone is bound by HBM with byte stores as well (0.300 ms) and keeps them.
            if (log2b >= 5u) {
                if (!__any_sync(0xffffffffu, changed)) continue;
                P x;
                source(x, p, t0, nvalid);
                uint32_t lo, hi;
                x.pack_exponents(lo, hi);
                const uint32_t top = __funnelshift_r(lo, hi, 8);  // bits 39:8
                const uint32_t before = __shfl_up_sync(0xffffffffu, top, 1);
                if (!changed) continue;
                const uint32_t rank = pre[kb >> 5] + __popc(word & ((1u << (kb & 31u)) - 1u));
                const uint32_t in_block = (t0 & ((1u << log2b) - 1u)) >> 3, a = in_block & 3u;
                uint32_t* const dst = reinterpret_cast<uint32_t*>(ti.pay_dst + base + payload_bytes_of_blocks<DT>(rank, log2b) +
                                                                  5u * (in_block - a)) + a;
                const uint32_t own = __funnelshift_l(before, lo, 8u * a);
                __stcs(dst, own);
                if (a == 3u) __stcs(dst + 1, top);
                uint32_t* const twin = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(dst) + tw.msg);
                __stcs(twin, own);
                if (a == 3u) __stcs(twin + 1, top);
                if (!CACHE) continue;
                x.template store_exp_full<Global>(ti.c_ptr + t0);
                x.template store_exp_full<Global>(ti.c_ptr + t0 + tw.cache);
                continue;
            }
        }
        if (!changed) continue;
        const uint32_t rank = pre[kb >> 5] + __popc(word & ((1u << (kb & 31u)) - 1u));
        uint8_t* cdst = ti.c_ptr + t0;
        P x;
        source(x, p, t0, nvalid);
        if constexpr (DT == CIERA_FP16) {
            // blocks of 16 values, short tiles: five packed bytes per piece (fewer for the last one), byte by byte
            uint8_t* pdst = ti.pay_dst + base + payload_bytes_of_blocks<DT>(rank, log2b) +
                            5u * ((t0 & ((1u << log2b) - 1u)) >> 3);
            uint32_t lo, hi;
            x.pack_exponents(lo, hi);
            const int nbytes = (5 * nvalid + 7) >> 3;
#pragma unroll
            for (int i = 0; i < 5; ++i)
                if (i < nbytes) put_byte<STEP>(pdst + i, (uint8_t)(i < 4 ? lo >> (8 * i) : hi), tw.msg);
            if (!CACHE) continue;
            if (nvalid == P::kValues) {
                x.template store_exp_full<Global>(cdst);
                if (STEP) x.template store_exp_full<Global>(cdst + tw.cache);
            } else {
                x.store_exp_partial(cdst, nvalid);
                if (STEP) x.store_exp_partial(cdst + tw.cache, nvalid);
            }
            continue;
        }
        uint8_t* pdst = ti.pay_dst + base + ((uint64_t)rank << log2b) + (t0 & ((1u << log2b) - 1u));
        if (nvalid == P::kValues) {
            x.template store_exp_full<Global>(pdst);
            if (CACHE) x.template store_exp_full<Global>(cdst);
            if (STEP) {
                x.template store_exp_full<Global>(pdst + tw.msg);
                if (CACHE) x.template store_exp_full<Global>(cdst + tw.cache);
            }
        } else {
            x.store_exp_partial(pdst, nvalid);
            if (CACHE) x.store_exp_partial(cdst, nvalid);
            if (STEP) {
                x.store_exp_partial(pdst + tw.msg, nvalid);
                if (CACHE) x.store_exp_partial(cdst + tw.cache, nvalid);
            }
        }
    }
}

// Sources of write_changed.  Of a stage in shared memory: new exponents or, LONG, the weights.
template <int DT, bool LONG>
__device__ __forceinline__ auto from_stage(const uint8_t* stage) {
    return [stage](Piece<DT>& x, int, uint32_t t0, int nvalid) {
        using P = Piece<DT>;
        if (LONG && nvalid != P::kValues) {
            x.split_first(stage + (size_t)t0 * Traits<DT>::kValueBytes, nvalid);
        } else if constexpr (LONG) {
            uint32_t w[P::kWeightWords];
            P::load_weights(stage + (size_t)t0 * Traits<DT>::kValueBytes, w);
            x.exponents_of(w);
        } else {
            x.template load_exp_full<Shared>(stage + t0);
        }
    };
}
// LONG: of the refreshed cache, where the same thread has put them (they are in L2 still), fetched ahead of the sending.
template <int DT>
struct FromCache {
    Piece<DT> x[Piece<DT>::kPerThread];
    __device__ __forceinline__ void fetch(const EncodeTileInfo& ti, uint32_t log2b, const uint32_t* bm, uint32_t tid) {
        using P = Piece<DT>;
#pragma unroll
        for (int p = 0; p < P::kPerThread; ++p) {
            const uint32_t t0 = P::start(tid, p), kb = t0 >> log2b;
            const int nvalid = piece_valid<DT>(t0, ti.nv);
            if (nvalid == 0 || !((bm[kb >> 5] >> (kb & 31u)) & 1u)) continue;
            if (nvalid == P::kValues)
                x[p].template load_exp_full<Global>(ti.c_ptr + t0);
            else
                x[p].load_exp_partial(ti.c_ptr + t0, nvalid);
        }
    }
    __device__ __forceinline__ void operator()(Piece<DT>& to, int p, uint32_t, int) const {
#pragma unroll
        for (int i = 0; i < Piece<DT>::kExpWords; ++i) to.e[i] = x[p].e[i];
    }
};

// STEP, fp32: one warp's 2 KB of reconstructed weights from the stage to global memory (one thread).
__device__ __forceinline__ void bulk_store_tile_part(const EncodeTileInfo& ti, const StepTwins& tw, const uint8_t* s_w,
                                                     uint32_t warp) {
    constexpr uint32_t kPart = (uint32_t)kTileValues * 4u / (uint32_t)kWarps;
    bulk_store(const_cast<uint8_t*>(ti.w_src) + tw.weights + (size_t)warp * kPart, s_w + (size_t)warp * kPart, kPart);
    bulk_commit();
}

// STEP, coarse blocks: the receiver's part of one tile.  Every consumer thread takes its pieces of the tile once
// more (the stage still holds the weights: sign and mantissa as they travel, and the exponents of changed blocks as
// they travel in the payload), puts the receiver's cached exponents of the unchanged blocks into their places and
// stores the reconstructed weights.  (Changed blocks: both caches are refreshed here, LONG, or by
// write_changed.)
// BULK: the thread's weights are left in their place of the stage instead.
template <int DT, bool FULL, bool BULK, bool LONG>
__device__ __forceinline__ void reconstruct(const EncodeTileInfo& ti, uint32_t log2b, const uint32_t* bm, uint8_t* s_w,
                                            const uint8_t* s_r, const StepTwins& tw, uint32_t tid) {
    using P = Piece<DT>;
    constexpr int VB = Traits<DT>::kValueBytes;
#pragma unroll
    for (int p = 0; p < P::kPerThread; ++p) {
        const uint32_t t0 = P::start(tid, p);
        const int nvalid = FULL ? (int)P::kValues : piece_valid<DT>(t0, ti.nv);
        if (nvalid == 0) continue;
        const uint32_t kb = t0 >> log2b;
        const bool changed = (bm[kb >> 5] >> (kb & 31u)) & 1u;
        uint8_t* const out = const_cast<uint8_t*>(ti.w_src) + tw.weights + (size_t)t0 * VB;
        const uint8_t* const r = ti.c_ptr + tw.cache + t0;
        uint32_t w[P::kWeightWords];
        if (!changed) {
            P x;
            if (ti.r_staged)
                x.template load_exp_full<Shared>(s_r + t0);
            else if (nvalid == P::kValues)
                x.template load_exp_full<Global>(r);
            else
                x.load_exp_partial(r, nvalid);
            x.exchange(s_w + (size_t)t0 * VB, w);
            if (BULK) P::template store_weights<Shared>(s_w + (size_t)t0 * VB, w);
        } else if (LONG || !BULK) {
            P::load_weights(s_w + (size_t)t0 * VB, w);
            if (LONG) {
                P x;
                x.exponents_of(w);
                uint8_t* const c = ti.c_ptr + t0;
                if (nvalid == P::kValues) {
                    x.template store_exp_full<Global>(c);
                    x.template store_exp_full<Global>(c + tw.cache);
                } else {
                    x.store_exp_partial(c, nvalid);
                    x.store_exp_partial(c + tw.cache, nvalid);
                }
            }
        }
        if (BULK) continue;
        if (nvalid == P::kValues)
            P::template store_weights<Global>(out, w);
        else
            P::store_weights_first(out, w, nvalid);
    }
}

// One block of B = 2^LB (fine) exponent bytes from shared memory to global memory; both addresses are B-aligned.
// (TWICE: and to the address `twin` bytes further on.)
template <int LB, bool TWICE>
__device__ __forceinline__ void copy_block(uint8_t* dst, const uint8_t* s_src, int64_t twin) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(s_src);
    if (LB == 0) {
        uint32_t v;
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
        __stcs(dst, (uint8_t)v);
        if (TWICE) __stcs(dst + twin, (uint8_t)v);
    } else if (LB == 1) {
        uint16_t v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
        __stcs(reinterpret_cast<uint16_t*>(dst), v);
        if (TWICE) __stcs(reinterpret_cast<uint16_t*>(dst + twin), v);
    } else if (LB == 2) {
        uint32_t v;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
        __stcs(reinterpret_cast<uint32_t*>(dst), v);
        if (TWICE) __stcs(reinterpret_cast<uint32_t*>(dst + twin), v);
    } else {
        const uint2 v = ld_shared8(s_src);
        st_stream8(dst, v);
        if (TWICE) st_stream8(dst + twin, v);
    }
}

// The same duty with fine blocks.  Here the work is split evenly over the tile's block flags
// rather than by pieces: thread t takes the flags of values [16 t, 16 t + 16) (16, 8, 4 or 2
// flags), walks the set ones and sends each flagged block's exponents to the payload (its rank
// = flags set before it in the tile).
// The cache is refreshed by whole 32-byte sectors instead: two neighbouring threads cover one sector of the
// tile's cached exponents, and if either of them has a changed block both store their 16 new exponents (the
// unchanged ones among them equal the cached ones).  A store of single changed bytes would leave the sector
// partly written in the L2 cache, to be completed from DRAM before it can be written back; whole sectors cost
// the same DRAM traffic and one store instruction per thread instead of one per changed value.
// (fp16: a changed block's exponents go out five bits each, the block rounded up to whole bytes -- 1, 2, 3 or 5
// bytes for 1, 2, 4 or 8 values -- and byte by byte, since such blocks start on any byte.)
// (STEP: the payload bytes also go to the received message.)
template <int DT, int LB, bool STEP>
__device__ __forceinline__ void write_changed_fine(const EncodeTileInfo& ti, const uint32_t* bm, const uint16_t* pre,
                                                   uint64_t base, const uint8_t* s_exp, const StepTwins& tw, uint32_t tid) {
    constexpr uint32_t B = 1u << LB;
    constexpr uint32_t kFlags = 16u >> LB;  // flags per thread
    const uint32_t bit0 = tid * kFlags;
    const uint32_t word = bm[bit0 >> 5], sh = bit0 & 31u;
    uint32_t bits = (word >> sh) & ((1u << kFlags) - 1u);  // never straddles a word
    const uint32_t v0 = tid * 16u;
    const uint32_t mine = bits != 0u ? 1u : 0u;
    if (mine | __shfl_xor_sync(0xffffffffu, mine, 1)) {
        if (v0 + 16u <= ti.nv) {
            st_stream16(ti.c_ptr + v0, ld_shared16(s_exp + v0));
        } else {
            for (uint32_t i = v0; i < ti.nv; ++i) ti.c_ptr[i] = s_exp[i];  // the unit's last values: never past its end
        }
    }
    if (bits == 0) return;
    const uint32_t rank = (uint32_t)pre[bit0 >> 5] + __popc(word & ((1u << sh) - 1u));
    if constexpr (DT == CIERA_FP16) {
        constexpr uint32_t kBlockBytes = (uint32_t)payload_bytes_of_blocks<DT>(1, LB);
        uint8_t* pdst = ti.pay_dst + base + (uint64_t)rank * kBlockBytes;
        while (bits) {
            const uint32_t j = (uint32_t)__ffs(bits) - 1u;
            bits &= bits - 1u;
            const uint32_t v = (bit0 + j) << LB;
            const uint32_t len = min(B, ti.nv - v);  // the unit's last block may be short
            unsigned long long packed = 0;
#pragma unroll
            for (uint32_t i = 0; i < B; ++i)
                if (i < len) packed |= (unsigned long long)(s_exp[v + i] & 31u) << (5u * i);
            const uint32_t nbytes = (5u * len + 7u) >> 3;
#pragma unroll
            for (uint32_t k = 0; k < kBlockBytes; ++k)
                if (k < nbytes) put_byte<STEP>(pdst + k, (uint8_t)(packed >> (8u * k)), tw.msg);
            pdst += kBlockBytes;
        }
        return;
    }
    uint8_t* pdst = ti.pay_dst + base + ((uint64_t)rank << LB);
    while (bits) {
        const uint32_t j = (uint32_t)__ffs(bits) - 1u;
        bits &= bits - 1u;
        const uint32_t v = (bit0 + j) << LB;  // the block's first value; < nv, since blocks past the end are never flagged
        if (ti.nv - v >= B) {
            copy_block<LB, STEP>(pdst, s_exp + v, tw.msg);
        } else {
            for (uint32_t i = 0; i < ti.nv - v; ++i) put_byte<STEP>(pdst + i, s_exp[v + i], tw.msg);  // the unit's short last block
        }
        pdst += B;
    }
}

// Bytes of shared memory in which one warp gathers the changed exponents of its 512 values before they go out:
// up to 15 bytes of skew in front (the gathered run starts at the same address modulo 16 as its place in the
// payload), up to 512 bytes, rounded up to whole 16-byte pieces.
constexpr uint32_t kWarpGatherBytes = 16u + 512u + 16u;
// FINE: for the changed exponents; fp16 with STEP: for the packed sign-plus-mantissa.
template <int DT, bool FINE, bool STEP>
constexpr uint32_t kGatherBytes = FINE ? kWarpGatherBytes : DT == CIERA_FP16 && STEP ? Piece<CIERA_FP16>::kWarpSmBytes : 0u;
// The gathering pays from about one changed exponent byte in four (measured with one value per block: 3.4 % changed
// 0.322 ms per layer gathered against 0.316 ms stored one by one, 50 % changed 0.429 against 0.548 ms; fp16, whole step,
// 40 % changed 0.795 against 1.18 ms; fp16's sender alone would gain 11 % there and lose 1-2 % with few changes).
constexpr uint32_t kGatherDensity = 4;

// Fine blocks, full tile.  A warp's 32 threads hold the flags of 512 consecutive values, so the changed blocks of
// the warp form one contiguous run of the unit's payload.  Instead of one scattered global store per changed
// block (measured: with one value per block and 3.4 % of the exponents changed, these byte stores cost more than
// a fifth of the kernel's time, with half of the exponents changed two thirds), the warp gathers the run in
// shared memory -- every thread walks its set flags as before, but stores into the warp's gather space -- and
// then writes it out in whole 16-byte pieces, one per lane, with single bytes only at the two ragged ends.
// The cache is refreshed by whole sectors as in write_changed_fine.
template <int DT, int LB, bool STEP>
__device__ __forceinline__ void write_changed_fine_full(const EncodeTileInfo& ti, const uint32_t* bm, const uint16_t* pre,
                                                        uint64_t base, const uint8_t* s_exp, uint8_t* s_gather,
                                                        const StepTwins& tw, uint32_t tid) {
    constexpr uint32_t kFlags = 16u >> LB;  // flags per thread
    constexpr uint32_t kBlockBytes = (uint32_t)payload_bytes_of_blocks<DT>(1, LB);
    const uint32_t lane = tid & 31u;
    const uint32_t bit0 = tid * kFlags;
    const uint32_t word = bm[bit0 >> 5], sh = bit0 & 31u;
    uint32_t bits = (word >> sh) & ((1u << kFlags) - 1u);  // never straddles a word
    const uint32_t v0 = tid * 16u;
    const uint32_t mine = bits != 0u ? 1u : 0u;
    if (mine | __shfl_xor_sync(0xffffffffu, mine, 1)) st_stream16(ti.c_ptr + v0, ld_shared16(s_exp + v0));
    // changed blocks of the tile before this thread's, before the warp's, and in the warp
    const uint32_t rank = (uint32_t)pre[bit0 >> 5] + __popc(word & ((1u << sh) - 1u));
    const uint32_t rank0 = __shfl_sync(0xffffffffu, rank, 0);
    const uint32_t total = __shfl_sync(0xffffffffu, rank + (uint32_t)__popc(bits), 31) - rank0;
    if (total == 0) return;
    uint8_t* const gdst = ti.pay_dst + base + (uint64_t)rank0 * kBlockBytes;  // where the warp's run goes
    const uint32_t skew = (uint32_t)(reinterpret_cast<uintptr_t>(gdst) & 15u);  // (not fp16: a multiple of the block size)
    uint8_t* out = s_gather + skew + (rank - rank0) * kBlockBytes;
    while (bits) {
        const uint32_t j = (uint32_t)__ffs(bits) - 1u;
        bits &= bits - 1u;
        const uint8_t* src = s_exp + ((bit0 + j) << LB);
        if (LB == 0) {
            *out = *src;
        } else if constexpr (DT == CIERA_FP16) {  // five bits each, the block rounded up to whole bytes
            unsigned long long packed = 0;
#pragma unroll
            for (uint32_t i = 0; i < (1u << LB); ++i) packed |= (unsigned long long)(src[i] & 31u) << (5u * i);
#pragma unroll
            for (uint32_t k = 0; k < kBlockBytes; ++k) out[k] = (uint8_t)(packed >> (8u * k));
        } else if (LB == 1) {
            *reinterpret_cast<uint16_t*>(out) = *reinterpret_cast<const uint16_t*>(src);
        } else if (LB == 2) {
            *reinterpret_cast<uint32_t*>(out) = *reinterpret_cast<const uint32_t*>(src);
        } else {
            st_shared8(out, ld_shared8(src));
        }
        out += kBlockBytes;
    }
    __syncwarp();
    // write-out: piece c covers bytes [16 c, 16 c + 16) of the gather space; the run occupies [skew, skew + len)
    // (the ragged ends byte by byte, one byte per lane; whole pieces in between, one per lane)
    const uint32_t end = skew + total * kBlockBytes;
    uint8_t* const g16 = gdst - skew;
    const uint32_t head_end = min((skew + 15u) & ~15u, end);  // first 16-byte boundary at or after the run's start
    const uint32_t tail_start = max(head_end, end & ~15u);     // last 16-byte boundary at or before its end
    if (skew + lane < head_end) put_byte<STEP>(g16 + skew + lane, s_gather[skew + lane], tw.msg);
    for (uint32_t c = ((skew + 15u) >> 4) + lane; 16u * c + 16u <= end; c += 32u) {
        const uint4 v = ld_shared16(s_gather + 16u * c);
        st_stream16(g16 + 16u * c, v);
        if (STEP) st_stream16(g16 + tw.msg + 16u * c, v);  // (the buffers lie a multiple of 16 bytes apart)
    }
    if (tail_start + lane < end) put_byte<STEP>(g16 + tail_start + lane, s_gather[tail_start + lane], tw.msg);
    __syncwarp();  // the gather space is free again
}

template <int DT, bool FINE, int HASH, bool STEP, bool LONG>
__device__ __forceinline__ void send_changed(const EncodeTileInfo& ti, uint32_t log2b, const uint32_t* bm,
                                             const uint16_t* pre, uint64_t base, uint32_t tile_payload_bytes,
                                             const uint8_t* s_exp, uint8_t* s_gather, const StepTwins& tw,
                                             uint32_t tid) {
    if (!FINE) {
        // (as in the consumers' main loop: the two instances named there keep the one form that tests as it goes)
        constexpr bool kOneBody = (DT == CIERA_BF16 && HASH == 0 && !STEP) || (DT == CIERA_FP32 && HASH != 0);
        if (!kOneBody && ti.nv == (uint32_t)kTileValues)
            write_changed<DT, HASH == 0 && !LONG, true, STEP, Share<DT, kConsumerWarps<DT, HASH>>>(ti, log2b, bm, pre, base, tw, tid,
                                                                                                from_stage<DT, LONG>(s_exp));
        else
            write_changed<DT, HASH == 0 && !LONG, false, STEP, Share<DT, kConsumerWarps<DT, HASH>>>(ti, log2b, bm, pre, base, tw, tid,
                                                                                                 from_stage<DT, LONG>(s_exp));
    } else if ((STEP || DT != CIERA_FP16) && ti.nv == (uint32_t)kTileValues && tile_payload_bytes >= (uint32_t)kTileValues / kGatherDensity) {
        // a full tile in which many exponents changed: gathered in shared memory, written out in whole pieces
        switch (log2b) {
            case 0: write_changed_fine_full<DT, 0, STEP>(ti, bm, pre, base, s_exp, s_gather, tw, tid); break;
            case 1: write_changed_fine_full<DT, 1, STEP>(ti, bm, pre, base, s_exp, s_gather, tw, tid); break;
            case 2: write_changed_fine_full<DT, 2, STEP>(ti, bm, pre, base, s_exp, s_gather, tw, tid); break;
            default: write_changed_fine_full<DT, 3, STEP>(ti, bm, pre, base, s_exp, s_gather, tw, tid); break;
        }
    } else {  // few changes (a store per changed block is cheaper than the gathering), a unit's last, short tile, or fp16's sender alone
        switch (log2b) {
            case 0: write_changed_fine<DT, 0, STEP>(ti, bm, pre, base, s_exp, tw, tid); break;
            case 1: write_changed_fine<DT, 1, STEP>(ti, bm, pre, base, s_exp, tw, tid); break;
            case 2: write_changed_fine<DT, 2, STEP>(ti, bm, pre, base, s_exp, tw, tid); break;
            default: write_changed_fine<DT, 3, STEP>(ti, bm, pre, base, s_exp, tw, tid); break;
        }
    }
}

// (The arguments stay within 160 bytes: with 168 a launch behind an event wait takes 0.4 us longer on the host; three small
// tables in a LayerPipeline 28.0 -> 29.3 us.)  per_tile: with STEP the list of tiles by address or null, with HASH `tile_hash`.
// `cache` is the sender's exponent cache or, with HASH, its HashCache; `tile_hash` (HASH only) gives
// the index of every tile's first block in it.
template <int DT, bool FINE, int HASH, bool STEP, bool LONG>
__global__ void __launch_bounds__(kEncodeThreads<DT, HASH>, kEncodeBlocksPerSM<DT, STEP>)
encode_kernel(const TileDesc* __restrict__ tiles, uint32_t n_tiles, const uint2* __restrict__ seq_runs, uint32_t n_runs,
              uint32_t spread_first, uint32_t clear_first, uint32_t log2b, const uint8_t* __restrict__ weights, uint8_t* cache, uint8_t* msgs,
              unsigned long long* wire_bytes, uint32_t* changed_blocks, void* status_words,
              void* scratch_a, unsigned int* scratch_b, int32_t* status,
              const void* __restrict__ per_tile, StepTwins tw, BufferEnds ends) {
    const uint32_t* const order = STEP ? static_cast<const uint32_t*>(per_tile) : nullptr;
    const unsigned long long* const tile_hash = HASH ? static_cast<const unsigned long long*>(per_tile) : nullptr;
    using Word = std::conditional_t<LONG, uint32_t, unsigned long long>;
    Word* const tile_status = static_cast<Word*>(status_words);
    // What lies behind the status words.  HASH: the counters and, an argument of its own, the count of finished blocks; else the
    // groups (LONG) and the counters.  (The time of the instances with HashCache follows how the compiler deals out their
    // registers, 70 to 77 in bf16 and fp16: with the others' arguments an OLMoE-shaped layer takes 306.4 us in bf16 and 426.8 in
    // fp16, like this, and with the first index into HashCache fetched together with the descriptor, 303.4 and 420.9.  fp32, 48
    // registers, fetches it later and counts the ring of results apart though it need not: half a layer in blocks of 16 657 ->
    // 641 us, of 64 292 -> 285, 2^23 values 25.9 -> 25.6.)
    constexpr bool kEarlyHash = HASH != 0 && DT != CIERA_FP32;
    constexpr bool kOwnCount = LONG || (HASH != 0 && DT == CIERA_FP32);
    unsigned long long* const groups = HASH ? nullptr : static_cast<unsigned long long*>(scratch_a);
    unsigned int* const counters = HASH ? static_cast<unsigned int*>(scratch_a) : scratch_b;
    unsigned int* const blocks_done = HASH ? scratch_b : scratch_b + 1;
    static_assert(!(HASH && FINE), "HashCache: blocks of 16 values and more");
    static_assert(!LONG || (STEP && !FINE), "long units: the whole step with coarse blocks");
    static_assert(!(HASH && STEP), "the whole step compares with the exponent cache");
    using P = Piece<DT>;
    constexpr int CW = kConsumerWarps<DT, HASH>;
    using S = Share<DT, CW>;
    constexpr int VB = Traits<DT>::kValueBytes;
    constexpr int SMB = Traits<DT>::kSmBytes;
    using Cfg = typename EncodeCfgOf<DT, FINE, HASH, STEP, LONG>::type;
    constexpr int SW = Cfg::kWStages;
    constexpr int SE = Cfg::kEStages;
    constexpr int SR = kResultStages<Cfg, LONG>;
    constexpr int kDefer = Cfg::kDefer;
    // coarse blocks: a tile's weights are reconstructed one slot after its votes, when its block flags are there
    constexpr bool kRebuild = STEP && !FINE;
    // fp32: the reconstructed weights of a full tile leave the stage by one bulk store per warp (64 bytes per lane
    // scatter over the stores of a warp)
    constexpr bool kBulkOut = STEP && DT == CIERA_FP32;
    static_assert(kDescRing > (LONG ? SW + SR : SE) + 2 && SR > kDefer && SR >= SW && (LONG || SE == SR), "ring depths");
    constexpr uint32_t kWBytes = kTileValues * VB;
    constexpr uint32_t kEBytes = kTileValues;
    extern __shared__ __align__(128) uint8_t smem[];
    uint8_t* const ring_w = smem;
    constexpr uint32_t kWStage = kWBytes + (STEP ? kEBytes : 0u);  // STEP: then the receiver's cached exponents
    uint8_t* const ring_e = smem + (size_t)SW * kWStage;
    using Ctl = EncodeCtl<SW, SE, SR, Cfg::kBmWords>;
    Ctl* ctl = reinterpret_cast<Ctl*>(ring_e + (size_t)SE * kEBytes);
    // HASH: per stage of the exponent ring, the tile's cached hashes and then the partial sums
    static_assert(sizeof(Ctl) % 16 == 0, "the hash stages follow the control block");
    static_assert(offsetof(Ctl, bm) % 16 == 0 && offsetof(Ctl, pre) % 4 == 0, "block flags are read 16 bytes at a time");
    uint8_t* const ring_h = reinterpret_cast<uint8_t*>(ctl) + sizeof(Ctl);
    const uint32_t kHoldBytes = HASH ? hash_hold_bytes<DT>(log2b) : 0u;
    const uint32_t kHStage = HASH ? kHoldBytes + hash_part_bytes<DT>(log2b) : 0u;

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const bool early_clear = spread_first < n_tiles && n_tiles - clear_first <= kEarlyClearTiles;
    volatile int* abort = &ctl->abort;
    // every consumer warp's gather space (in place of the hash stages)
    uint8_t* const s_gather = ring_h + (size_t)(warp < (uint32_t)CW ? warp : 0u) * kGatherBytes<DT, FINE, STEP>;

    if (tid == 0) {
        for (int s = 0; s < SW; ++s) {
            mbar_init(&ctl->full_w[s], 1);
            mbar_init(&ctl->empty_w[s], CW);
        }
        for (int s = 0; s < SE; ++s) {
            mbar_init(&ctl->full_e[s], 1);
            mbar_init(&ctl->empty_e[s], CW);
        }
        for (int s = 0; s < SR; ++s) {
            mbar_init(&ctl->voted[s], CW);
            mbar_init(&ctl->summed[s], 1);
            mbar_init(&ctl->resolved[s], 1);
        }
        ctl->abort = 0;
        ctl->issued = 0;
        ctl->seen = 0;
        mbar_fence_init();
    }
    // The producer fetches its first tile's descriptor before it waits for the kernel before this one, which cannot be writing
    // the plan's tables (see pdl_wait): one round trip less in front of the first loads.  Whole step back to back, fetched
    // behind the wait / before it: one matrix of 524 288 values on 4 shards, bf16 6.68 / 6.53 us, fp32 9.21 / 8.91; one expert
    // on 16 shards 20.39 / 20.20; registers and spills of all instances are the same.
    TileDesc nxt;
    unsigned long long hb_nxt = 0;  // HASH: index of the tile's first block in HashCache
    if (tid == 32u * (uint32_t)CW) {
        const uint32_t first = first_tile<STEP>(seq_runs, order, n_runs, spread_first, n_tiles, blockIdx.x);
        if (first != kNoTile) {
            nxt = load_tile_desc(tiles + first);
            if (kEarlyHash) hb_nxt = __ldg(tile_hash + first);
        }
    }
    pdl_wait();
    __syncthreads();

    // The block's tiles form a sequence k = 0, 1, 2, ... that only the producer knows in advance;
    // it closes the sequence with kResolvers end markers (one for each resolver warp), which the
    // other roles pass on to each other through the same barriers as real tiles.
    if (warp == (uint32_t)CW) {
        // ---------------------------------------------------------------- producer
        if (lane == 0) {
            TileWalk<STEP, LONG> walk(seq_runs, order, counters, n_runs, spread_first, n_tiles, gridDim.x, blockIdx.x);
            uint32_t seq_nxt = 0;
            uint32_t tile_nxt = walk.next(seq_nxt);  // (descriptors are fetched one tile ahead, the first one above)
            if (HASH && !kEarlyHash && tile_nxt != kNoTile) hb_nxt = __ldg(tile_hash + tile_nxt);
            uint32_t markers = 0;
            for (uint32_t k = 0;; ++k) {
                const TileDesc td = nxt;
                const uint32_t tile = tile_nxt;
                const uint32_t seq = seq_nxt;
                const unsigned long long hb = hb_nxt;
                auto fetch = [&]() {
                    tile_nxt = walk.next(seq_nxt);
                    if (tile_nxt != kNoTile) {
                        nxt = load_tile_desc(tiles + tile_nxt);
                        if (HASH) hb_nxt = __ldg(tile_hash + tile_nxt);
                    }
                };
                const bool late = walk.late();
                if (tile != kNoTile && !late) fetch();
                const uint32_t sw = k % SW, se = k % SE;
                if (k >= (uint32_t)SW && !mbar_wait(&ctl->empty_w[sw], ((k / SW) & 1u) ^ 1u, abort, status)) break;
                if (k >= (uint32_t)SE && !mbar_wait(&ctl->empty_e[se], ((k / SE) & 1u) ^ 1u, abort, status)) break;
                ctl->tile_idx[k % kDescRing] = tile;
                if (tile == kNoTile) {  // end marker
                    mbar_arrive(&ctl->full_w[sw]);
                    if (HASH) mbar_arrive(&ctl->full_e[se]);
                    if (++markers == (uint32_t)kResolvers) break;
                    continue;
                }
                // (What the others need is written before the copies are started: the other way round the descriptor and its flags stay
                // live across them, which no instance of 48 registers has room for.  Spill stores / loads 16 / 8 -> 36 / 16 bytes and
                // an OLMoE-shaped layer 277 -> 296 us, bf16 sender; whole step on one tensor of 2^28 values 28 / 24 -> 100 / 76, 399 -> 415;
                // sender with HashCache 306 -> 313.)
                ctl->desc[k % kDescRing] = td;
                ctl->seq[k % kDescRing] = seq;
                const uint64_t v0 = (uint64_t)td.tile_in_unit * kTileValues;
                const uint64_t left = td.n_unit - v0;
                bool r_staged = true;
                {
                    const uint64_t smoff = sm_offset(td.n_unit, log2b);
                    EncodeTileInfo ti;
                    ti.sm_dst = msgs + td.msg_off + smoff + sm_bytes_of_values<DT>(v0);
                    ti.pay_dst = msgs + td.msg_off + smoff + pad16(sm_section_bytes(td.n_unit, DT));
                    ti.c_ptr = HASH ? cache + hb * 16ull : cache + td.c_off;
                    ti.w_src = weights + td.w_off;
                    ti.nv = (uint32_t)min((uint64_t)kTileValues, left);
                    // Only unchanged blocks need the receiver's cached exponents.  Where the tile one ring of stages
                    // before was dense (see kDenseValues) they are not staged: with every block changed that is 1 byte
                    // of 12 per value that need not be read.
                    r_staged = FINE || k < (uint32_t)(LONG ? SW : SE) ||
                               ctl->agg[LONG ? (k - SW) % SR : se] < payload_bytes_of_blocks<DT>(kDenseValues >> log2b, log2b);
                    ti.r_staged = r_staged ? 1u : 0u;
                    ctl->info[k % kDescRing] = ti;
                }
                // A unit's last, short tile is staged too, in whole 16-byte pieces; the consumers drop what lies behind its
                // last value.  Only behind the last value of a whole buffer there need not be anything.
                const uint32_t nvt = (uint32_t)min((uint64_t)kTileValues, left);
                const uint32_t w_bytes = (nvt * (uint32_t)VB + 15u) & ~15u, e_bytes = (nvt + 15u) & ~15u;
                if (ends.has(tile, nvt)) {
                    stage_buffer_end(ring_w + (size_t)sw * kWStage, weights + td.w_off, nvt * (uint32_t)VB,
                                     HASH ? nullptr : ring_e + (size_t)se * kEBytes, cache + td.c_off, nvt,
                                     STEP && r_staged ? kWBytes : 0u, tw.cache, &ctl->full_w[sw]);
                } else if (HASH) {
                    mbar_arrive_expect_tx(&ctl->full_w[sw], w_bytes);
                    bulk_load(ring_w + (size_t)sw * kWStage, weights + td.w_off, w_bytes, &ctl->full_w[sw]);
                } else {
                    // all copies of the tile complete on the one barrier the consumers wait for
                    mbar_arrive_expect_tx(&ctl->full_w[sw], w_bytes + e_bytes + (STEP && r_staged ? e_bytes : 0u));
                    bulk_load(ring_w + (size_t)sw * kWStage, weights + td.w_off, w_bytes, &ctl->full_w[sw]);
                    bulk_load(ring_e + (size_t)se * kEBytes, cache + td.c_off, e_bytes, &ctl->full_w[sw]);
                    if (STEP && r_staged)
                        bulk_load(ring_w + (size_t)sw * kWStage + kWBytes, cache + tw.cache + td.c_off, e_bytes,
                                  &ctl->full_w[sw]);
                }
                if constexpr (HASH) {
                    // the cached hashes of the tile's blocks (16 bytes each)
                    const uint32_t nblk = (nvt + (1u << log2b) - 1u) >> log2b;
                    mbar_arrive_expect_tx(&ctl->full_e[se], nblk * 16u);
                    bulk_load(ring_h + (size_t)se * kHStage, cache + hb * 16ull, nblk * 16u, &ctl->full_e[se]);
                }
                ctl->issued = k + 1;
                if (late) fetch();
            }
            cp_async_wait_all();  // (an aborted run: none in flight when the block ends)
        }
    } else if (warp == (uint32_t)CW + 1u) {
        // ---------------------------------------------------------------- aggregator
        uint64_t run_incl = 0;  // payload bytes of the current alone-worked unit up to the last tile
        uint32_t byte_acc = 0;  // its bitmap byte in the making (tiles of fewer than 8 blocks)
        uint32_t markers = 0;
        for (uint32_t k = 0;; ++k) {
            const uint32_t se = k % SE, sr = k % SR;
            if (!mbar_wait(&ctl->voted[sr], (k / SR) & 1u, abort, status)) break;
            const uint32_t tile = ctl->tile_idx[k % kDescRing];
            if (tile == kNoTile) {  // pass the end marker on to the resolver in charge of slot k
                if (lane == 0) mbar_arrive(&ctl->summed[sr]);
                if (++markers == (uint32_t)kResolvers) break;
                continue;
            }
            const TileDesc td = ctl->desc[k % kDescRing];
            const uint32_t seq_bits = ctl->seq[k % kDescRing];
            const bool seq = seq_bits != 0;
            HashTile ht{nullptr, nullptr, nullptr};
            if constexpr (HASH) {
                // the cached hashes were staged by a bulk copy that completes on full_e: observe it here too
                if (!mbar_wait(&ctl->full_e[se], (k / SE) & 1u, abort, status)) break;
                ht.hold = reinterpret_cast<const ulonglong2*>(ring_h + (size_t)se * kHStage);
                ht.part = reinterpret_cast<const ulonglong2*>(ring_h + (size_t)se * kHStage + kHoldBytes);
                ht.dst = reinterpret_cast<ulonglong2*>(ctl->info[k % kDescRing].c_ptr);
            }
            const uint32_t nbt = kTileValues >> log2b;
            const uint32_t nv = (uint32_t)min((uint64_t)kTileValues, td.n_unit - (uint64_t)td.tile_in_unit * kTileValues);
            const uint32_t nblk = (nv + (1u << log2b) - 1u) >> log2b;
            const bool last = td.tile_in_unit == td.n_tiles_unit - 1u;
            uint8_t* const msg = msgs + td.msg_off;
            uint8_t* const bitmap_dst = msg + (uint64_t)td.tile_in_unit * (nbt >> 3);
            const uint64_t agg = aggregate_tile<DT, FINE, HASH>(td, tile, log2b, !seq, ctl->ballot[sr], ctl->bm[sr], ctl->pre[sr],
                                                                tile_status, groups, ht, nv, lane);
            uint64_t excl = 0;
            if (seq) {
                // the run is this block's: the tile's offset is the running sum; a run that does not start its
                // unit carries on from the inclusive offset that the run before it left in its last tile's
                // status word (that run went out many draws earlier; the wait is bounded all the same; reading
                // the word in the producer thread instead, tiles ahead, was slower)
                excl = run_incl;
                if (td.tile_in_unit == 0)
                    excl = 0;
                else if (seq_bits & kSeqRunStart) {
                    excl = wait_status(tile_status + tile - 1, status) & (LONG ? (Word)kShortValueMask : (Word)kValueMask);
                    __syncwarp();
                    if (lane == 0) st_status(tile_status + tile - 1, (Word)0);  // its one reader leaves the word empty again
                }
                run_incl = excl + agg;
                if ((seq_bits & kSeqRunEnd) && !last && lane == 0)
                    st_status(tile_status + tile, (LONG ? (Word)kShortPrefix : (Word)kFlagPrefix) | (Word)run_incl);
            }
            // What the others wait for goes out before the tile's bitmap and the unit's totals: the chain votes - sums -
            // offset - sending is what small tables wait for.  The flags that are still needed are in registers by then, since
            // the stage may be refilled.  (Whole step of 4736 units of 67 values 45 -> 41 us, sender with 64 values per block
            // 0.281 -> 0.274 ms per OLMoE-shaped layer; with HashCache the other order is the faster one for small tables.  So it is for
            // the sender alone on 2-byte values where a block has four spread tiles and more to work through: one unit of
            // 10^8 bf16 values 109.8 -> 107.5 us, 35 of 688 745 fp16 values 38.7 -> 37.4, 64 of 2 097 152 bf16 values 142 -> 138;
            // fp32, two of 30 000 001, 108 -> 111.)
            uint32_t word = 0;
            if (FINE)
                store_bitmap_fine<STEP>(bitmap_dst, ctl->bm[sr], nblk, tw, lane);
            else if (32u * lane < nbt)
                word = ctl->bm[sr][lane];
            auto report = [&]() {
                if (!FINE && nbt >= 8) store_bitmap<STEP>(bitmap_dst, word, nblk, tw, lane);
                if (!seq) return;
                if (nbt < 8) {
                    const uint32_t tpb = 8u / nbt, p = td.tile_in_unit & (tpb - 1u);
                    byte_acc = (p == 0 ? 0u : byte_acc) | (word << (p * nbt));  // (lane 0)
                    if ((p == tpb - 1u || last) && lane == 0)
                        put_byte<STEP>(msg + td.tile_in_unit / tpb, (uint8_t)byte_acc, tw.msg);
                }
                if (last) finish_unit<DT, STEP>(td, log2b, run_incl, msgs, tw.msg, wire_bytes, changed_blocks, lane);
            };
            const bool report_first = HASH != 0 || (!STEP && DT != CIERA_FP32 && !seq && n_tiles - spread_first >= 4u * gridDim.x);
            if (report_first) report();
            if (lane == 0) {
                if (seq) ctl->base[sr] = excl;
                ctl->agg[sr] = agg;
            }
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&ctl->summed[sr]);
                if (seq) mbar_arrive(&ctl->resolved[sr]);
            }
            if (!report_first) report();
        }
    } else if (warp >= (uint32_t)CW + 2u) {
        // ---------------------------------------------------------------- resolvers (slots k = i, i + R, ...)
        for (uint32_t k = warp - ((uint32_t)CW + 2u);; k += kResolvers) {
            const uint32_t sr = k % SR;
            if (!mbar_wait(&ctl->summed[sr], (k / SR) & 1u, abort, status)) break;
            const uint32_t tile = ctl->tile_idx[k % kDescRing];
            if (tile == kNoTile) {
                if (early_clear) {
                    // this warp looks back no more; the last one of the grid empties the status words
                    uint32_t last = 0;
                    if (lane == 0) {
                        __threadfence();
                        last = atomicAdd(blocks_done, 1u) + 1u == gridDim.x * (uint32_t)kResolvers ? 1u : 0u;
                    }
                    if (__shfl_sync(0xffffffffu, last, 0)) {
                        __threadfence();
                        clear_status(tile_status, groups, clear_first, n_tiles, lane, 32u);
                        if (lane == 0) atomicExch(blocks_done, 0u);
                    }
                }
                break;
            }
            if (ctl->seq[k % kDescRing] != 0) continue;  // the aggregator has done it all
            const TileDesc td = ctl->desc[k % kDescRing];
            resolve_tile<DT, STEP>(td, tile, log2b, ctl->agg[sr], ctl->bm[sr], msgs, tw.msg, wire_bytes, changed_blocks,
                                   tile_status, groups, status, lane, [&](uint64_t excl) {
                                       if (lane == 0) {
                                           ctl->base[sr] = excl;
                                           mbar_arrive(&ctl->resolved[sr]);
                                       }
                                   });
        }
    } else {
        // ---------------------------------------------------------------- consumers
        uint32_t k_end = kNoTile;  // slot of the first end marker, once seen
        uint32_t k = 0;
        // stage and phase of slot k in the rings, and of slot k - kDefer in the ring of results, kept
        // as running counters (the ring depths are no powers of two)
        uint32_t sw = 0, pw = 0, se = 0, pe = 0, sr_own = 0, je = 0, pj = 0;
        uint32_t& sr = kOwnCount ? sr_own : se;  // stage of slot k in the ring of results: the ring of exponents is as long, but for LONG
        uint32_t rw = 0, rr = 0, pr = 0;  // kRebuild: stages of slot k - 1 in the rings of weights and results, phase in the latter
        // HASH: the lanes of a warp that share a block (a power of two, at most the warp) add up their terms
        const uint32_t hash_lanes_l2 = min(5u, log2b - (uint32_t)P::kLog2Values);
        for (;; ++k) {
            // LONG: a spread tile is sent kDefer slots later, from the cache: its exponents are fetched here
            std::conditional_t<LONG, FromCache<DT>, int> ahead;
            bool deferred = false;
            if constexpr (LONG) {
                deferred = k >= (uint32_t)kDefer && k - kDefer < k_end && ctl->seq[(k - kDefer) % kDescRing] == 0;
                if (deferred) ahead.fetch(ctl->info[(k - kDefer) % kDescRing], log2b, ctl->bm[je], tid);
            }
            // (the producer starts the loads of slot k only once both of its stages are free, and the cached
            // exponents land on the same barrier as the weights; with HashCache the cached hashes, which only
            // the aggregator reads, land on full_e)
            if (!mbar_wait(&ctl->full_w[sw], pw, abort, status)) break;
            if (tid == 0) ctl->seen = k + 1;
            const bool marker = ctl->tile_idx[k % kDescRing] == kNoTile;
            if (marker) {
                if (k_end == kNoTile) k_end = k;
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&ctl->voted[sr]);  // pass the end marker on to the aggregator
                    mbar_arrive(&ctl->empty_w[sw]);  // and hand the marker's (unused) stages back
                    mbar_arrive(&ctl->empty_e[se]);
                }
            } else {
                const EncodeTileInfo ti = ctl->info[k % kDescRing];
                const uint32_t nv = ti.nv;
                uint8_t* const s_w = ring_w + (size_t)sw * kWStage;
                const uint8_t* const s_r = s_w + kWBytes;  // STEP: the receiver's cached exponents
                uint8_t* const s_e = ring_e + (size_t)se * kEBytes;
                uint64_t hash_a[S::kPerThread], hash_b[S::kPerThread];  // HASH: the pieces' sums of terms
                // The pieces of this thread.  Most instances compile the loop twice: for full tiles (staged
                // in shared memory, every piece complete, no tests on the way) and for a unit's last, short
                // tile; that measured 2-12 % faster (fp16 most).  Two instances keep one loop that tests as it
                // goes, which measured faster for them: bf16 with coarse blocks and the exponent cache (1 %),
                // fp32 with HashCache (5 %).
                constexpr bool kOneBody = (DT == CIERA_BF16 && !FINE && HASH == 0 && !STEP) || (DT == CIERA_FP32 && HASH != 0);
                if constexpr (kOneBody) {
                    // a plain loop that tests as it goes
#define CIERA_PIECES_FULL false
#define CIERA_PIECES_WHOLE (nv == (uint32_t)kTileValues)
#include "ciera_encode_pieces.inc"
#undef CIERA_PIECES_FULL
#undef CIERA_PIECES_WHOLE
                } else {
                    auto pieces = [&](auto full_tag) {
                        constexpr bool kFull = decltype(full_tag)::value;
#define CIERA_PIECES_FULL kFull
#define CIERA_PIECES_WHOLE kFull
#include "ciera_encode_pieces.inc"
#undef CIERA_PIECES_FULL
#undef CIERA_PIECES_WHOLE
                    };
                    if (nv == (uint32_t)kTileValues)
                        pieces(std::true_type{});
                    else
                        pieces(std::false_type{});
                }
                if constexpr (HASH) {
                    uint64_t* const part = reinterpret_cast<uint64_t*>(ring_h + (size_t)se * kHStage + kHoldBytes);
                    if constexpr (HASH == 3) {
                        // the tile's cached hashes have to be there now (they land on full_e)
                        if (!mbar_wait(&ctl->full_e[se], pe, abort, status)) break;
                        finish_hash_groups<DT, S::kPerThread>(hash_a, hash_b, hash_lanes_l2, log2b, nv, tid,
                                                              reinterpret_cast<const uint64_t*>(ring_h + (size_t)se * kHStage),
                                                              reinterpret_cast<uint64_t*>(ti.c_ptr),
                                                              reinterpret_cast<uint8_t*>(part), lane);
                    } else if constexpr (S::kPerThread == 4) {
                        reduce_hash_rows(hash_a, hash_b, hash_lanes_l2, log2b, S::start(tid, 0), part, lane);
                    } else {
                        reduce_hash_terms<S::kPerThread>(hash_a, hash_b, hash_lanes_l2, (S::start(tid, 0) >> P::kLog2Values) >> hash_lanes_l2,
                                                         (S::start(tid, S::kPerThread - 1) >> P::kLog2Values) >> hash_lanes_l2, part, lane);
                    }
                }
                if (kBulkOut && !kRebuild) fence_async_shared();  // the reconstructed weights, before lane 0's bulk store reads them
                __syncwarp();  // the warp's shared-memory accesses above are ordered before lane 0's arrives
                if (lane == 0) {
                    mbar_arrive(&ctl->voted[sr]);
                    if (LONG) mbar_arrive(&ctl->empty_e[se]);
                    if (!kRebuild) {
                        if (kBulkOut && nv == (uint32_t)kTileValues) {
                            bulk_store_tile_part(ti, tw, s_w, warp);
                            bulk_wait_read<0>();
                        }
                        mbar_arrive(&ctl->empty_w[sw]);
                    }
                }
            }
            if constexpr (kRebuild) {
                // the receiver's part of the tile before this one: its block flags are there by now
                if (k != 0 && k - 1u < k_end) {
                    if (!mbar_wait(&ctl->summed[rr], pr, abort, status)) break;
                    const EncodeTileInfo ti = ctl->info[(k - 1u) % kDescRing];
                    uint8_t* const s_w = ring_w + (size_t)rw * kWStage;
                    const bool full = ti.nv == (uint32_t)kTileValues;
                    if (full)
                        reconstruct<DT, true, kBulkOut, LONG>(ti, log2b, ctl->bm[rr], s_w, s_w + kWBytes, tw, tid);
                    else
                        reconstruct<DT, false, false, LONG>(ti, log2b, ctl->bm[rr], s_w, s_w + kWBytes, tw, tid);
                    if (kBulkOut) fence_async_shared();
                    __syncwarp();
                    if (kBulkOut && full && lane == 0) bulk_store_tile_part(ti, tw, s_w, warp);
                    if (LONG && ctl->seq[(k - 1u) % kDescRing] != 0) {  // a tile of a run: its offset came with its flags
                        send_changed<DT, FINE, HASH, STEP, LONG>(ti, log2b, ctl->bm[rr], ctl->pre[rr], ctl->base[rr],
                                                                 (uint32_t)ctl->agg[rr], s_w, s_gather, tw, tid);
                        __syncwarp();
                    }
                    if (lane == 0) {
                        if (kBulkOut && full) bulk_wait_read<0>();
                        mbar_arrive(&ctl->empty_w[rw]);
                    }
                }
                if (k != 0) {
                    if (++rw == (uint32_t)SW) rw = 0;
                    if (++rr == (uint32_t)SR) {
                        rr = 0;
                        pr ^= 1u;
                    }
                }
            }

            // the changed exponents of the tile handled kDefer slots ago: its offset is known by now
            if (k >= (uint32_t)kDefer) {
                if constexpr (LONG) {
                    if (deferred) {
                        if (!mbar_wait(&ctl->resolved[je], pj, abort, status)) break;
                        const EncodeTileInfo ti = ctl->info[(k - kDefer) % kDescRing];
                        if (ti.nv == (uint32_t)kTileValues)
                            write_changed<DT, false, true, STEP, S>(ti, log2b, ctl->bm[je], ctl->pre[je], ctl->base[je], tw, tid, ahead);
                        else
                            write_changed<DT, false, false, STEP, S>(ti, log2b, ctl->bm[je], ctl->pre[je], ctl->base[je], tw, tid, ahead);
                    }
                } else if (k - kDefer < k_end) {
                    if (!mbar_wait(&ctl->resolved[je], pj, abort, status)) break;
                    send_changed<DT, FINE, HASH, STEP, false>(ctl->info[(k - kDefer) % kDescRing], log2b, ctl->bm[je], ctl->pre[je],
                                                        ctl->base[je], (uint32_t)ctl->agg[je], ring_e + (size_t)je * kEBytes,
                                                        s_gather, tw, tid);
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->empty_e[je]);
                }
                if (++je == (uint32_t)SR) {
                    je = 0;
                    pj ^= 1u;
                }
            }
            if (marker && k + 1u == k_end + (uint32_t)kResolvers) break;  // that was the last end marker
            if (++sw == (uint32_t)SW) {
                sw = 0;
                pw ^= 1u;
            }
            if (++se == (uint32_t)SE) {
                se = 0;
                pe ^= 1u;
            }
            if (kOwnCount && ++sr == (uint32_t)SR) sr = 0;
        }
        // tiles whose changed exponents are still to be sent (when kDefer > kResolvers)
        if (!*abort && k_end != kNoTile) {
            for (uint32_t j = k + 1u >= (uint32_t)kDefer ? k + 1u - kDefer : 0u; j < k_end; ++j) {
                const uint32_t je = j % SR;
                if (LONG && ctl->seq[j % kDescRing] != 0) continue;  // sent already
                if (!mbar_wait(&ctl->resolved[je], (j / SR) & 1u, abort, status)) break;
                const EncodeTileInfo ti = ctl->info[j % kDescRing];
                if constexpr (LONG) {
                    if (j + (uint32_t)SW < k_end) {
                        FromCache<DT> ahead;
                        ahead.fetch(ti, log2b, ctl->bm[je], tid);
                        write_changed<DT, false, false, STEP, S>(ti, log2b, ctl->bm[je], ctl->pre[je], ctl->base[je], tw, tid, ahead);
                        continue;
                    }
                }
                // (LONG: the weights stage has not been filled again)
                send_changed<DT, FINE, HASH, STEP, LONG>(ti, log2b, ctl->bm[je], ctl->pre[je], ctl->base[je], (uint32_t)ctl->agg[je],
                                                         LONG ? ring_w + (size_t)(j % SW) * kWStage : ring_e + (size_t)je * kEBytes,
                                                         s_gather, tw, tid);
                __syncwarp();
                if (!LONG && lane == 0) mbar_arrive(&ctl->empty_e[je]);
            }
        }
    }

    if (kBulkOut) bulk_wait_all<0>();  // this thread's bulk stores are complete before the block ends
    // leave together; after an aborted run wait (bounded) for bulk copies that are still in flight
    __syncthreads();
    if (tid == 0 && ctl->abort) {
        for (uint32_t k = ctl->seen; k < ctl->issued; ++k) {
            for (uint32_t i = 0; i < kMaxBarrierPolls; ++i)
                if (mbar_try_wait(&ctl->full_w[k % SW], (k / SW) & 1u)) break;
            if (HASH) {
                for (uint32_t i = 0; i < kMaxBarrierPolls; ++i)
                    if (mbar_try_wait(&ctl->full_e[k % SE], (k / SE) & 1u)) break;
            }
        }
    }
    // The scratch is handed back the way it was found, all zero: the hand-off words of the runs were emptied by
    // their readers, the run counter by its last draw; the status words of the spread tiles (read by any number
    // of later tiles) and the counter of finished blocks are emptied by whoever finishes last.  Where the words are
    // few that is the resolver warp that looks back last, while the consumers still send (a fence and an atomic
    // behind everything else cost the smallest tables more than a microsecond); where they are many it is the
    // block that finishes last, with all its threads.  Without spread tiles there is nothing to empty.
    // (clear_first: a step in parts leaves the status words to the parts that follow, and the last part empties all)
    if (early_clear || spread_first >= n_tiles) return;
    __shared__ unsigned int s_last;
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(blocks_done, 1u) + 1u == gridDim.x ? 1u : 0u;
    }
    __syncthreads();
    if (s_last) {
        __threadfence();
        clear_status(tile_status, groups, clear_first, n_tiles, tid, (uint32_t)kEncodeThreads<DT, HASH>);
        if (tid == 0) atomicExch(blocks_done, 0u);
    }
}

// (with HashCache the size depends on the block size: see hash_hold_bytes, hash_part_bytes)
template <int DT, bool FINE, int HASH, bool STEP, bool LONG>
static size_t encode_smem_bytes(uint32_t log2b) {
    using Cfg = typename EncodeCfgOf<DT, FINE, HASH, STEP, LONG>::type;
    constexpr int SW = Cfg::kWStages, SE = Cfg::kEStages;
    const size_t hash_stage = HASH ? (size_t)hash_hold_bytes<DT>(log2b) + hash_part_bytes<DT>(log2b) : 0;
    // the SM's 228 KB hold that many blocks, with the 1 KB each that the system takes
    static_assert(HASH || kEncodeBlocksPerSM<DT, STEP> *
                                  ((size_t)SW * kTileValues * (Traits<DT>::kValueBytes + (STEP ? 1 : 0)) + (size_t)SE * kTileValues +
                                   sizeof(EncodeCtl<SW, SE, kResultStages<Cfg, LONG>, Cfg::kBmWords>) + (size_t)kWarps * kGatherBytes<DT, FINE, STEP> + 1024) <=
                              233472,
                  "thread blocks per SM");
    return (size_t)SW * kTileValues * (Traits<DT>::kValueBytes + (STEP ? 1 : 0)) + (size_t)SE * kTileValues +
           sizeof(EncodeCtl<SW, SE, kResultStages<Cfg, LONG>, Cfg::kBmWords>) + (size_t)SE * hash_stage + (size_t)kWarps * kGatherBytes<DT, FINE, STEP>;
}

// Largest grid whose blocks are all resident at once, per device and block size (0 = not yet known).
template <int DT, bool FINE, int HASH, bool STEP, bool LONG>
static int encode_grid_limit(uint32_t log2b, int* out) {
    static std::atomic<int> cached[64][16];  // (zero-initialised; any host thread may be the first to fill an entry)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda_error(e);
    if (dev < 0 || dev >= 64 || log2b >= 16) return CIERA_ERR_UNSUPPORTED;
    if (cached[dev][log2b].load(std::memory_order_acquire) == 0) {
        const size_t smem = encode_smem_bytes<DT, FINE, HASH, STEP, LONG>(log2b);
        // (the limit set here is the largest any block size asks for: the smallest block of the class)
        e = cudaFuncSetAttribute(encode_kernel<DT, FINE, HASH, STEP, LONG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)encode_smem_bytes<DT, FINE, HASH, STEP, LONG>(FINE ? 0u : HASH == 1 ? kHashShortRingsLog2 + 1u : kFineLog2));
        if (e != cudaSuccess) return record_cuda_error(e);
        int per_sm = 0, sms = 0, coop = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, encode_kernel<DT, FINE, HASH, STEP, LONG>, kEncodeThreads<DT, HASH>, smem);
        if (e != cudaSuccess) return record_cuda_error(e);
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return record_cuda_error(e);
        e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
        if (e != cudaSuccess) return record_cuda_error(e);
        if (per_sm < 1 || sms < 1 || !coop) return CIERA_ERR_UNSUPPORTED;
        cached[dev][log2b].store(per_sm * sms, std::memory_order_release);
    }
    *out = cached[dev][log2b].load(std::memory_order_acquire);
    return CIERA_OK;
}

// `scratch`: the status words (and, LONG, the groups' words), then the counters of runs, of finished blocks and of spread tiles
// (see workspace_groups_offset); all zero when the kernel starts, and all zero again when it has finished without a
// device-side error.
// part of a step: the tiles at places [lo, hi) of `order` (null: table order), all of them spread; the last part empties
// the status words
struct EncodePart {
    const uint32_t* order;
    uint32_t lo, hi;
    bool last;
};
template <int DT, bool FINE, int HASH = 0, bool STEP = false, bool LONG = false>
static int launch_encode(const ciera_plan* p, const void* weights_dev, void* sender_cache_dev, void* messages_dev,
                         uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, void* scratch, int32_t* status_dev,
                         cudaStream_t s, StepTwins tw = StepTwins{0, 0, 0}, const EncodePart* part = nullptr) {
    int limit = 0;
    const int rc = encode_grid_limit<DT, FINE, HASH, STEP, LONG>(p->log2b, &limit);
    if (rc) return rc;
    const TileDesc* tiles = p->tiles_dev;
    const uint32_t all_tiles = (uint32_t)p->tiles.size();
    uint32_t nt = part ? part->hi : all_tiles;
    const uint32_t to_do = part ? part->hi - part->lo : all_tiles;
    const uint32_t grid = to_do < (uint32_t)limit ? to_do : (uint32_t)limit;
    const uint2* seq_runs = p->seq_runs_dev;
    const bool spread_all = part || p->spread_all;
    uint32_t n_runs = spread_all ? 0u : (uint32_t)p->seq_runs.size();
    uint32_t spread_first = part ? part->lo : spread_all ? 0u : p->seq_first.back();
    uint32_t clear_first = !part ? spread_first : part->last ? 0u : nt;
    uint32_t log2b = p->log2b;
    const uint8_t* w = (const uint8_t*)weights_dev;
    uint8_t* c = (uint8_t*)sender_cache_dev;
    uint8_t* m = (uint8_t*)messages_dev;
    unsigned long long* wb = (unsigned long long*)wire_bytes_dev;
    unsigned long long* groups = (unsigned long long*)((uint8_t*)scratch + workspace_groups_offset(all_tiles));
    unsigned int* counters = (unsigned int*)((uint8_t*)scratch + workspace_sender_counters_offset(all_tiles));
    void* scratch_a = HASH ? static_cast<void*>(counters) : groups;
    unsigned int* scratch_b = HASH ? counters + 1 : counters;
    const void* per_tile = HASH ? static_cast<const void*>(p->tile_hash_dev) : part ? part->order : nullptr;
    const size_t smem = encode_smem_bytes<DT, FINE, HASH, STEP, LONG>(log2b);
    BufferEnds ends{p->weights_end_tile, HASH ? kNoTile : p->cache_end_tile, p->several_end_tiles};
    const bool has_spread = spread_first < nt;  // look-back between blocks
    // With a tile to a block and nothing else a tile looks back at blocks before its own only, so the blocks need not all be
    // resident and the launch may begin while the kernel before it drains -- provided that blocks start in the order of their
    // numbers, which the hardware does and the programming model does not promise (the runs of short units rest on it too: a
    // block's first two are given by its number).  Were a block to start after one that waits for it, with all SMs taken by
    // other kernels for longer than the bound on the wait, the step would end with CIERA_ERR_TIMEOUT, not hang.  Drawing the
    // tile from a counter instead costs a round trip before the first load: 64 tiles 6.6 -> 7.0 us.  (Two or three neighbouring
    // tiles to a block would keep that for more tables; measured on whole steps back to back: 384 tiles 15.3 us against
    // 14.1 with a cooperative launch and every grid-th tile, 768 tiles 18.3 against 20.1, 1024 tiles in fours 30.1 against 25.0.)
    const bool one_each = n_runs == 0 && to_do <= grid;
    cudaError_t e;
    if (has_spread && !one_each) {
        // cooperative launch: the runtime starts the grid only when all of its blocks fit on the
        // GPU together, which is what the look-back between blocks relies on
        void* args[] = {&tiles, &nt, &seq_runs, &n_runs, &spread_first, &clear_first, &log2b, &w, &c, &m, &wb,
                        &changed_blocks_dev, &scratch, &scratch_a, &scratch_b, &status_dev, &per_tile, &tw, &ends};
        e = cudaLaunchCooperativeKernel((const void*)encode_kernel<DT, FINE, HASH, STEP, LONG>, dim3(grid), dim3(kEncodeThreads<DT, HASH>), args,
                                        smem, s);
    } else {
        e = launch_after(encode_kernel<DT, FINE, HASH, STEP, LONG>, dim3(grid), kEncodeThreads<DT, HASH>, smem, s, tiles, nt, seq_runs, n_runs,
                         spread_first, clear_first, log2b, w, c, m, wb, changed_blocks_dev, scratch, scratch_a, scratch_b, status_dev,
                         per_tile, tw, ends);
    }
    if (e != cudaSuccess) return record_cuda_error(e);
    count_launch();
    return CIERA_OK;
}

// picks the kernel for the plan's precision and block class
template <int DT>
static int launch_encode_of(const ciera_plan* p, const void* weights_dev, void* sender_cache_dev, void* messages_dev,
                            uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, void* scratch, int32_t* status_dev,
                            cudaStream_t s, const StepTwins* tw, const EncodePart* part) {
    if (tw && !is_fine(p->log2b) && p->long_units)
        return launch_encode<DT, false, 0, true, true>(p, weights_dev, sender_cache_dev, messages_dev, wire_bytes_dev, changed_blocks_dev,
                                                       scratch, status_dev, s, *tw, part);
    auto launch = [&](auto fine, auto step) {
        return launch_encode<DT, decltype(fine)::value, 0, decltype(step)::value>(
            p, weights_dev, sender_cache_dev, messages_dev, wire_bytes_dev, changed_blocks_dev, scratch, status_dev, s,
            tw ? *tw : StepTwins{0, 0, 0}, part);
    };
    if (is_fine(p->log2b)) return tw ? launch(std::true_type{}, std::true_type{}) : launch(std::true_type{}, std::false_type{});
    return tw ? launch(std::false_type{}, std::true_type{}) : launch(std::false_type{}, std::false_type{});
}
// (tw: the whole step; null: the sender's part alone)
static int launch_encode_any(const ciera_plan* p, const void* weights_dev, void* sender_cache_dev, void* messages_dev,
                             uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, void* scratch, int32_t* status_dev,
                             cudaStream_t s, const StepTwins* tw = nullptr, const EncodePart* part = nullptr) {
    auto* launch = p->dtype == CIERA_FP16   ? launch_encode_of<CIERA_FP16>
                   : p->dtype == CIERA_BF16 ? launch_encode_of<CIERA_BF16>
                                            : launch_encode_of<CIERA_FP32>;
    return launch(p, weights_dev, sender_cache_dev, messages_dev, wire_bytes_dev, changed_blocks_dev, scratch, status_dev, s,
                  tw, part);
}

// the sender with HashCache: blocks of 16 values and more (checked by the caller)
int launch_encode_hashed(const ciera_plan* p, const void* weights_dev, void* hash_cache_dev, void* messages_dev,
                         uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, void* scratch, int32_t* status_dev,
                         cudaStream_t s) {
    const bool short_rings = p->log2b <= kHashShortRingsLog2;
    if (p->dtype == CIERA_BF16 && hash_finished_by_consumers<CIERA_BF16>(p->log2b))
        return launch_encode<CIERA_BF16, false, 3>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                   changed_blocks_dev, scratch, status_dev, s);
    if (p->dtype == CIERA_FP16 && hash_finished_by_consumers<CIERA_FP16>(p->log2b))
        return launch_encode<CIERA_FP16, false, 3>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                   changed_blocks_dev, scratch, status_dev, s);
    if (p->dtype == CIERA_FP16)
        return short_rings ? launch_encode<CIERA_FP16, false, 2>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                                 changed_blocks_dev, scratch, status_dev, s)
                           : launch_encode<CIERA_FP16, false, 1>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                                 changed_blocks_dev, scratch, status_dev, s);
    if (p->dtype == CIERA_FP32 && hash_finished_by_consumers<CIERA_FP32>(p->log2b))
        return launch_encode<CIERA_FP32, false, 3>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                   changed_blocks_dev, scratch, status_dev, s);
    if (p->dtype == CIERA_BF16)
        return short_rings ? launch_encode<CIERA_BF16, false, 2>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                                 changed_blocks_dev, scratch, status_dev, s)
                           : launch_encode<CIERA_BF16, false, 1>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                                 changed_blocks_dev, scratch, status_dev, s);
    return short_rings ? launch_encode<CIERA_FP32, false, 2>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                             changed_blocks_dev, scratch, status_dev, s)
                       : launch_encode<CIERA_FP32, false, 1>(p, weights_dev, hash_cache_dev, messages_dev, wire_bytes_dev,
                                                             changed_blocks_dev, scratch, status_dev, s);
}

}  // namespace ciera

using namespace ciera;

static bool misaligned16(const void* p) { return ((uintptr_t)p & 15u) != 0; }

extern "C" int ciera_encode(const ciera_plan* p, const void* weights_dev, void* sender_cache_dev, void* messages_dev,
                            uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, void* workspace_dev,
                            int32_t* status_dev, void* stream) {
    if (!p) return CIERA_ERR_INVALID_ARG;
    if (!p->tiles.empty() && !p->tiles_dev) return CIERA_ERR_NOT_BOUND;
    if (p->n_units == 0) return CIERA_OK;
    if (!wire_bytes_dev || !changed_blocks_dev) return CIERA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const uint32_t nt = (uint32_t)p->tiles.size();
    cudaError_t e;
    if (p->has_empty_units) {  // units without tiles: their outputs are written here
        e = cudaMemsetAsync(wire_bytes_dev, 0, sizeof(uint64_t) * p->n_units, s);
        if (e != cudaSuccess) return record_cuda_error(e);
        e = cudaMemsetAsync(changed_blocks_dev, 0, sizeof(uint32_t) * p->n_units, s);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    if (nt == 0) return CIERA_OK;
    if (!weights_dev || !sender_cache_dev || !messages_dev || !workspace_dev) return CIERA_ERR_INVALID_ARG;
    if (misaligned16(weights_dev) || misaligned16(sender_cache_dev) || misaligned16(messages_dev) ||
        misaligned16(workspace_dev) || ((uintptr_t)wire_bytes_dev & 7u) || ((uintptr_t)changed_blocks_dev & 3u))
        return CIERA_ERR_MISALIGNED;
    // scratch = one look-back status word per tile, then the counters: all zero on entry (ciera_workspace_init,
    // or left so by the previous call, a step with other words among them), and the kernel hands it back all zero
    return launch_encode_any(p, weights_dev, sender_cache_dev, messages_dev, wire_bytes_dev, changed_blocks_dev,
                             workspace_dev, status_dev, s);
}

static StepTwins step_twins(const void* weights, const void* sender_cache, const void* msg_send, const void* msg_recv,
                            const void* receiver_cache, const void* weights_out) {
    return StepTwins{(int64_t)((intptr_t)msg_recv - (intptr_t)msg_send),
                     (int64_t)((intptr_t)receiver_cache - (intptr_t)sender_cache),
                     (int64_t)((intptr_t)weights_out - (intptr_t)weights)};
}

// One launch reads and writes all buffers of a step side by side.  Three calls in a row only need what is live between
// them: the reconstructed weights may go to where the weights lay a little further on, or to where the message was sent
// from.  Here, each buffer has to have its place to itself, but for weights that are reconstructed in place (the same
// bytes, tile by tile, unless units share theirs).
bool ciera::step_buffers_apart(const ciera_plan* p, const void* weights, const void* sender_cache, const void* msg_send,
                               const void* msg_recv, const void* receiver_cache, const void* weights_out) {
    struct {
        uintptr_t at;
        uint64_t bytes;
    } const r[6] = {{(uintptr_t)weights, p->weights_extent},  {(uintptr_t)weights_out, p->weights_extent},
                    {(uintptr_t)sender_cache, p->cache_extent}, {(uintptr_t)receiver_cache, p->cache_extent},
                    {(uintptr_t)msg_send, p->msg_extent},       {(uintptr_t)msg_recv, p->msg_extent}};
    for (int i = 0; i < 6; ++i)
        for (int j = i + 1; j < 6; ++j) {
            if (i == 0 && j == 1 && weights == weights_out && p->by_address_ok) continue;
            if (r[i].at < r[j].at + r[j].bytes && r[j].at < r[i].at + r[i].bytes) return false;
        }
    return true;
}

// The checks of a step, and the outputs of units without tiles.
int ciera::step_begin(const ciera_plan* p, const void* weights_dev, const void* sender_cache_dev, const void* msg_send_dev,
                            const void* msg_recv_dev, const void* receiver_cache_dev, const void* weights_out_dev,
                            uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev, const void* workspace_dev, cudaStream_t s) {
    if (!p) return CIERA_ERR_INVALID_ARG;
    if (!p->tiles.empty() && !p->tiles_dev) return CIERA_ERR_NOT_BOUND;
    if (p->n_units == 0) return CIERA_OK;
    if (!wire_bytes_dev || !changed_blocks_dev) return CIERA_ERR_INVALID_ARG;
    if (p->has_empty_units) {  // units without tiles: their outputs are written here
        cudaError_t e = cudaMemsetAsync(wire_bytes_dev, 0, sizeof(uint64_t) * p->n_units, s);
        if (e != cudaSuccess) return record_cuda_error(e);
        e = cudaMemsetAsync(changed_blocks_dev, 0, sizeof(uint32_t) * p->n_units, s);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    if (p->tiles.empty()) return CIERA_OK;
    if (!weights_dev || !sender_cache_dev || !msg_send_dev || !msg_recv_dev || !receiver_cache_dev || !weights_out_dev ||
        !workspace_dev)
        return CIERA_ERR_INVALID_ARG;
    if (misaligned16(weights_dev) || misaligned16(sender_cache_dev) || misaligned16(msg_send_dev) ||
        misaligned16(msg_recv_dev) || misaligned16(receiver_cache_dev) || misaligned16(weights_out_dev) ||
        misaligned16(workspace_dev) || ((uintptr_t)wire_bytes_dev & 7u) || ((uintptr_t)changed_blocks_dev & 3u))
        return CIERA_ERR_MISALIGNED;
    return CIERA_OK;
}

extern "C" int ciera_step(const ciera_plan* p, const void* weights_dev, void* sender_cache_dev, void* msg_send_dev,
                          void* msg_recv_dev, void* receiver_cache_dev, void* weights_out_dev, uint64_t* wire_bytes_dev,
                          uint32_t* changed_blocks_dev, void* workspace_dev, int32_t* status_dev, void* stream) {
    cudaStream_t s = (cudaStream_t)stream;
    const int rc = step_begin(p, weights_dev, sender_cache_dev, msg_send_dev, msg_recv_dev, receiver_cache_dev,
                                    weights_out_dev, wire_bytes_dev, changed_blocks_dev, workspace_dev, s);
    if (rc || p->tiles.empty()) return rc;
    if (!step_buffers_apart(p, weights_dev, sender_cache_dev, msg_send_dev, msg_recv_dev, receiver_cache_dev, weights_out_dev)) {
        int r = ciera_encode(p, weights_dev, sender_cache_dev, msg_send_dev, wire_bytes_dev, changed_blocks_dev, workspace_dev,
                             status_dev, stream);
        if (r == CIERA_OK) r = ciera_transport(p, msg_send_dev, msg_recv_dev, wire_bytes_dev, workspace_dev, status_dev, stream);
        if (r == CIERA_OK)
            r = ciera_decode(p, msg_recv_dev, receiver_cache_dev, weights_out_dev, wire_bytes_dev, workspace_dev, status_dev, stream);
        return r;
    }
    const StepTwins tw = step_twins(weights_dev, sender_cache_dev, msg_send_dev, msg_recv_dev, receiver_cache_dev, weights_out_dev);
    return launch_encode_any(p, weights_dev, sender_cache_dev, msg_send_dev, wire_bytes_dev, changed_blocks_dev,
                             workspace_dev, status_dev, s, &tw);
}

// (the caller has checked the buffers as ciera_step does)
int ciera::launch_step_part(const ciera_plan* p, const ciera_device_buffers* b, uint32_t lo, uint32_t hi, cudaStream_t s) {
    const StepTwins tw = step_twins(b->weights_dev, b->sender_cache_dev, b->msg_send_dev, b->msg_recv_dev,
                                    b->receiver_cache_dev, b->weights_out_dev);
    const EncodePart part{p->tiles_by_address_dev, lo, hi, hi == (uint32_t)p->tiles.size()};
    return launch_encode_any(p, b->weights_dev, b->sender_cache_dev, b->msg_send_dev, b->wire_bytes_dev,
                             b->changed_blocks_dev, b->workspace_dev, b->status_dev, s, &tw, &part);
}

// ------------------------------------------------------------------------------------------
// Encode for callers that have no scratch buffer to give.
//
// Some callers hand this library only the buffers they already own -- parameter shards, caches,
// communication buffers -- and cannot come up with one more device allocation at the moment of the
// call: a training runtime whose memory pool has claimed the whole GPU (a fresh allocation would
// fail or fragment the pool), a gather hook that must not synchronise the device (allocating
// does), a plug-in that was given pointers but no allocator.  For them the look-back scratch of
// the encode kernel lives in the library itself: a fixed array in device memory that every GPU
// loading the library holds from load until the process exits.

static __device__ __align__(256) unsigned long long g_encode_scratch[CIERA_NOALLOC_MAX_TILES + 2];

// Device address of g_encode_scratch on the current device.  In host code the array's name is only
// a handle for the runtime, not an address a kernel could use, so the address is looked up once
// per device (with that device current) and kept.
static int encode_scratch_address(unsigned long long** out) {
    static std::atomic<unsigned long long*> cached[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda_error(e);
    if (dev < 0 || dev >= 64) return CIERA_ERR_UNSUPPORTED;
    unsigned long long* ptr = cached[dev].load(std::memory_order_acquire);
    if (ptr == nullptr) {
        void* q = nullptr;
        e = cudaGetSymbolAddress(&q, g_encode_scratch);
        if (e != cudaSuccess) return record_cuda_error(e);
        if (q == nullptr) return CIERA_ERR_CUDA;
        ptr = static_cast<unsigned long long*>(q);
        cached[dev].store(ptr, std::memory_order_release);
    }
    *out = ptr;
    return CIERA_OK;
}

extern "C" int ciera_encode_noalloc(const ciera_plan* p, const void* weights_dev, void* sender_cache_dev,
                                    void* messages_dev, uint64_t* wire_bytes_dev, uint32_t* changed_blocks_dev,
                                    int32_t* status_dev, void* stream) {
    if (!p) return CIERA_ERR_INVALID_ARG;
    if (!p->tiles.empty() && !p->tiles_dev) return CIERA_ERR_NOT_BOUND;
    const uint32_t nt = (uint32_t)p->tiles.size();
    if (nt > CIERA_NOALLOC_MAX_TILES) return CIERA_ERR_TOO_LARGE;
    if (p->n_units == 0) return CIERA_OK;
    if (!wire_bytes_dev || !changed_blocks_dev) return CIERA_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    if (p->has_empty_units) {  // units without tiles: their outputs are written here
        e = cudaMemsetAsync(wire_bytes_dev, 0, sizeof(uint64_t) * p->n_units, s);
        if (e != cudaSuccess) return record_cuda_error(e);
        e = cudaMemsetAsync(changed_blocks_dev, 0, sizeof(uint32_t) * p->n_units, s);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    if (nt == 0) return CIERA_OK;
    if (!weights_dev || !sender_cache_dev || !messages_dev) return CIERA_ERR_INVALID_ARG;
    if (misaligned16(weights_dev) || misaligned16(sender_cache_dev) || misaligned16(messages_dev) ||
        ((uintptr_t)wire_bytes_dev & 7u) || ((uintptr_t)changed_blocks_dev & 3u))
        return CIERA_ERR_MISALIGNED;
    unsigned long long* scratch = nullptr;
    int rc = encode_scratch_address(&scratch);
    if (rc) return rc;
    // the array keeps what the previous call left in it: the status words of this call's tiles and
    // the unit counter behind them have to start at zero
    e = cudaMemsetAsync(scratch, 0, sizeof(unsigned long long) * nt + 16, s);
    if (e != cudaSuccess) return record_cuda_error(e);
    return launch_encode_any(p, weights_dev, sender_cache_dev, messages_dev, wire_bytes_dev, changed_blocks_dev, scratch,
                             status_dev, s);
}
