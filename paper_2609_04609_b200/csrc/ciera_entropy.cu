// Entropy stage (paper Section 3.1; Algorithm 1: payload <- ANSEncode(...), newExp <- ANSDecode(...)):
// the exponents of changed blocks are coded with rANS between the sender step and the transport, and
// decoded between the transport and the receiver step.  The paper uses a vendor library whose
// stream format is not public; the coder and the layout here are this library's own.
//
// Model: one static table per unit, 256 symbols, probabilities in 1/4096 (f[s] = max(1,
// floor(h[s] * 4096 / P)) for the symbols that occur; a shortfall goes to the most frequent symbol,
// an excess is taken from the largest entries).
// Coder: 32-bit state x in [2^16, 2^32), 16-bit words.
//   encode s:  if x >= f[s] * 2^20: emit x mod 2^16, x >>= 16;   x <- (x / f) * 4096 + x mod f + c[s]
//   decode:    slot = x mod 4096, s = symbol of slot;  x <- f[s] * (x / 4096) + slot - c[s];
//              if x < 2^16: x <- x * 2^16 + next word
// The raw payload is cut into segments of 4096 bytes; one warp codes a segment with its 32 lanes as
// 32 interleaved coders (lane l owns bytes 32 t + l).  The encoder walks the steps t backwards and
// appends the words its lanes emit (ballot, rank = lanes below); the decoder walks forwards and
// takes the words from the end of the list backwards, so neither side needs per-lane streams.
// Coded section: [A x u16 f] [n_seg x u32 word counts] [segments: 32 x u32 final states, words,
// 2 zero bytes if the count is odd].  It replaces the raw payload only if strictly shorter; the
// receiver knows the raw length from the bitmap and so tells the two forms apart by the length.
// The symbols are the exponents of the changed blocks (Algorithm 1 codes {exp[k] | bitmap[k] = 1}):
// for bf16 and fp32 the payload's bytes as they are, A = 256 table entries.  For fp16 the five-bit
// packing of the payload is undone into a scratch first (one symbol per byte, A = 32 entries travel),
// segments are cut every 4096 symbols, "raw length" above is the packed payload's, and the receiver
// packs the decoded symbols back into the message.
//
// Work split: a unit of up to 64 segments' worth of values (262 144) is done by one thread block from
// start to end (histogram, model, segments into a scratch, coded form into the message).  Longer
// units go through a chain of launches whose grids run over chunks of 64 segments, so that their
// work spreads over the GPU: sender = histogram, model, segments, layout, copy; receiver = layout,
// segments, restore.  Nothing waits for another thread block anywhere.
#include <type_traits>

#include "ciera_bits.cuh"

namespace ciera {

constexpr uint32_t kProbBits = 12, kProbScale = 1u << kProbBits;
constexpr uint32_t kRansL = 1u << 16;
constexpr uint32_t kSegment = 4096;                              // bytes of raw payload per segment
constexpr uint32_t kSegWordsMax = kSegment * kProbBits / 16;     // 3072: a symbol adds at most 12 bits
constexpr uint32_t kSegSlot = 4 * 32 + 2 * kSegWordsMax;         // 6272 bytes: states + words
constexpr int kEntThreads = 256, kEntWarps = kEntThreads / 32;
// A unit's thread block has kEntThreads threads where there are units enough to fill the GPU, else kEntMiddle (two blocks
// to an SM) or kEntWide (one), as long as all of them are resident at once: a segment is a serial chain of 128 steps
// (about 8 us), and a block codes as many segments at a time as it has warps.  Sender's / receiver's stage, us: four units
// of 32 segments 66 / 92 with 8 warps, 32 / 31 with 32; 160 units of 32 slots, 7 of them in use, 41 / 62 with 8 warps, 27 / 33
// with 16 (cut into several blocks each: 42 / 54), all in use 100 / 127 and 64 / 65 (cut: 55 / 60); 288 units of 32 slots, 7
// in use, 47 / 66 and 30 / 33.  Whole step with the stage, 192 units of 8 segments: 79 with 8 warps, 107 with 32.
constexpr int kEntWide = 1024, kEntMiddle = 512;
constexpr uint32_t kLongSegs = kEntLongSlots;  // units with more segment slots than this take the chunked path

__host__ __device__ inline uint64_t segments_of(uint64_t bytes) { return (bytes + kSegment - 1) / kSegment; }
__host__ __device__ inline uint32_t segment_bytes(uint32_t nw) { return 4u * 32u + 2u * nw + ((nw & 1u) ? 2u : 0u); }
// bytes of the frequency table that travels: one u16 per symbol of the alphabet
__host__ __device__ inline uint32_t model_bytes(int dt) { return dt == CIERA_FP16 ? 64u : 512u; }

// ---------------------------------------------------------------------------------- shared pieces

// Adds the bytes pay[lo, hi) to the warp-private histograms (lo a multiple of 16, pay 16-byte aligned).
template <int T>
__device__ __forceinline__ void histogram_add(uint32_t (*hist)[256], const uint8_t* pay, uint64_t lo, uint64_t hi,
                                              uint32_t tid) {
    const uint32_t warp = tid >> 5;
    for (uint64_t i = lo + (uint64_t)tid * 16; i < hi; i += (uint64_t)T * 16) {
        if (i + 16 <= hi) {
            const uint4 v = *reinterpret_cast<const uint4*>(pay + i);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 16; ++k) atomicAdd(&hist[warp][(w[k >> 2] >> (8 * (k & 3))) & 0xFFu], 1u);
        } else {
            for (uint64_t k = i; k < hi; ++k) atomicAdd(&hist[warp][pay[k]], 1u);
        }
    }
}

// Exclusive running sums of f[0..255] by one warp (lane l owns symbols 8 l .. 8 l + 7): returns the sum of
// the symbols before the lane's first one and leaves the sums inside its group in local[]; `total`
// gets the sum of all.
__device__ __forceinline__ uint32_t warp_prefix256(const uint16_t* f, uint32_t lane, uint32_t local[8], uint32_t& total) {
    uint32_t run = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        local[i] = run;
        run += f[8 * lane + i];
    }
    uint32_t incl = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += t;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - run;
}

// Index of the largest of v[0..255], the lowest index among equals (one warp; v(s) gives the value).
template <class V>
__device__ __forceinline__ uint32_t warp_argmax256(V v, uint32_t lane) {
    unsigned long long key = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t s = 8 * lane + i;
        const unsigned long long k = ((unsigned long long)v(s) << 8) | (255u - s);
        key = k > key ? k : key;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, o);
        key = k > key ? k : key;
    }
    return 255u - (uint32_t)(key & 255u);
}

// Frequencies from counts (h[256] in shared memory, P = their sum): thread s owns symbol s, then the
// first warp settles the sum.  Ends with a barrier; f is then final.
__device__ __forceinline__ void normalise_model(const uint32_t* h, uint64_t P, uint16_t* f, uint32_t tid) {
    if (tid < 256u) {
        uint32_t v = 0;
        if (h[tid]) {
            v = P < (1ull << 20) ? h[tid] * kProbScale / (uint32_t)P : (uint32_t)((uint64_t)h[tid] * kProbScale / P);
            if (v == 0) v = 1;
        }
        f[tid] = (uint16_t)v;
    }
    __syncthreads();
    if (tid < 32) {
        uint32_t local[8], sum;
        warp_prefix256(f, tid, local, sum);
        if (sum < kProbScale) {  // the shortfall goes to the most frequent symbol
            const uint32_t best = warp_argmax256([&](uint32_t s) { return h[s]; }, tid);
            if (tid == 0) f[best] = (uint16_t)(f[best] + (kProbScale - sum));
        } else {  // an excess is taken from the largest entries
            uint32_t excess = sum - kProbScale;
            while (excess) {
                const uint32_t big = warp_argmax256([&](uint32_t s) { return (uint32_t)f[s]; }, tid);
                const uint32_t take = min((uint32_t)f[big] - 1u, excess);
                __syncwarp();
                if (tid == 0) f[big] = (uint16_t)(f[big] - take);
                __syncwarp();
                excess -= take;
            }
        }
    }
    __syncthreads();
}

// The coder's tables from final frequencies.  Ends with a barrier.
// q = x / f for x < f * 2^20 <= 2^32 is one 32-bit multiplication and a shift.  With s = floor(log2 f), P = 2^(32 + s),
// m = floor(P / f) and e = (m + 1) * f - P:
//   f = 1                     m = 2^32 - 1 gives x - 1 (x > 0), the missing 1 * (4096 - f) goes into c
//   f a power of two          m = 2^31, shift s - 1
//   f * 2^20 * e <= P         q = ((m + 1) * x) / P, the round-up reciprocal (all f < 2^11, most others; Granlund and
//                             Montgomery, Division by Invariant Integers using Multiplication, 1994)
//   else                      q = (m * (x + 1)) / P, the round-down one (Robison, N-Bit Unsigned Division via N-Bit
//                             Multiply-Add, 2005): exact if f * 2^20 * (f - e) <= P, which follows from
//                             e > P / (f * 2^20) >= 2^23 / f for 2^11 < f < 2^12
// At most one symbol is of the last kind; whether there is one comes back (the same in all threads).  An entry of 16
// bytes holds what a coder step needs:
//   {multiplier, largest x below f * 2^20, c, (4096 - f) << 5 | shift, bit 31: x + 1}
__device__ __forceinline__ bool encoder_tables(const uint16_t* f, uint4* enc, uint32_t tid) {
    const uint32_t fs = tid < 256u && f[tid] ? f[tid] : 1u;
    uint32_t s = 31u - (uint32_t)__clz(fs), m = 0xFFFFFFFFu, plus = 0u;
    if (fs & (fs - 1u)) {
        // floor(2^(32 + s) / f) in two 32-bit divisions: s + 16 < 28 and the first remainder is below 2^12
        const uint32_t a = 1u << (s + 16u), q1 = a / fs, r1 = (a - q1 * fs) << 16, q0 = r1 / fs;
        m = (q1 << 16) + q0;
        const uint32_t e = fs - (r1 - q0 * fs);  // (m + 1) * f - P
        if (((unsigned long long)fs << 20) * e <= (1ull << (32u + s)))
            m += 1u;
        else
            plus = 1u;
    } else if (s) {
        m = 0x80000000u;
        s -= 1u;
    }
    if (tid < 256u) {
        enc[tid].x = m;
        enc[tid].y = (uint32_t)(((unsigned long long)fs << 20) - 1ull);
        enc[tid].w = ((kProbScale - fs) << 5) | s | (plus << 31);
    }
    if (tid < 32) {
        uint32_t local[8], total;
        const uint32_t base = warp_prefix256(f, tid, local, total);
#pragma unroll
        for (int i = 0; i < 8; ++i) enc[8 * tid + i].z = base + local[i] + (f[8 * tid + i] == 1 ? kProbScale - 1u : 0u);
    }
    return __syncthreads_or((int)plus) != 0;
}

// One warp codes one segment: src[0, n) -> slot (32 states, then the words).  Returns the word count.
// Bound by instruction issue.  A lane's symbols lie 32 bytes apart; four steps' worth of a warp (128 bytes) come in
// with one load, a word per lane, and are turned into a word of four successive symbols per lane by a 4 x 4
// transposition inside every quad of lanes (two exchanges, two byte permutes).  Sixteen steps are loaded ahead of the
// sixteen in work.  (With a staged copy of the segment, a byte load per step and a 64-bit reciprocal: 0.180 ms per
// OLMoE-shaped layer, B = 512, q = 0.22; like this 0.154.  4 / 6 thread blocks per SM instead of 5: 0.168 / 0.190.)
// `src` is 4-byte aligned.  PLUS: the tables hold a symbol whose quotient takes x + 1.
template <bool PLUS>
__device__ __forceinline__ uint32_t encode_segment(const uint8_t* src, uint32_t n, const uint4* enc, uint8_t* slot,
                                                   uint32_t lane) {
    uint16_t* const words = reinterpret_cast<uint16_t*>(slot + 4 * 32);
    uint32_t x = kRansL, nw = 0;
    const uint32_t below = (1u << lane) - 1u;
    // one coder step of this lane for symbol s
    auto step = [&](uint32_t s, bool has) {
        const uint4 en = enc[s];
        const bool emit = has && x > en.y;  // x >= f * 2^20
        const uint32_t votes = __ballot_sync(0xffffffffu, emit);
        if (emit) {
            words[nw + __popc(votes & below)] = (uint16_t)x;
            x >>= 16;
        }
        nw += __popc(votes);
        // x / f (the shift takes the low 5 bits of its amount), then q * 4096 + x mod f + c
        const uint32_t q = __funnelshift_r(__umulhi(PLUS ? x + (en.w >> 31) : x, en.x), 0u, en.w);
        const uint32_t y = x + en.z + q * (PLUS ? (en.w >> 5) & 0x1FFFu : en.w >> 5);
        x = has ? y : x;
    };
    // the rows of 32 symbols behind the last whole block of 16 rows come first (the coder walks backwards)
    const uint32_t blocks = n >> 9;
    for (uint32_t t = (n + 31u) >> 5; t-- > 16u * blocks;) {
        const uint32_t at = 32u * t + lane;
        step(at < n ? src[at] : 0u, at < n);
    }
    if (blocks) {
        // lane 4 c + j loads row j of a group of four rows, columns 4 c .. 4 c + 3
        const uint32_t* from = reinterpret_cast<const uint32_t*>(src) + 128u * (blocks - 1u) + 8u * (lane & 3u) + (lane >> 2);
        const uint32_t sel1 = (lane & 1u) ? 0x3715u : 0x6240u, sel2 = (lane & 2u) ? 0x3276u : 0x5410u;
        uint32_t next[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) next[i] = from[32 * i];
        for (uint32_t b = blocks; b != 0u;) {
            uint32_t cur[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) cur[i] = next[i];
            from -= 128;
            if (--b) {
#pragma unroll
                for (int i = 0; i < 4; ++i) next[i] = from[32 * i];
            }
#pragma unroll
            for (int i = 3; i >= 0; --i) {
                uint32_t v = cur[i];
                v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 1), sel1);
                v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 2), sel2);
                step(v >> 24, true);
                step(__byte_perm(v, 0u, 0x4442u), true);
                step(__byte_perm(v, 0u, 0x4441u), true);
                step(v & 0xFFu, true);
            }
        }
    }
    reinterpret_cast<uint32_t*>(slot)[lane] = x;
    if (lane == 0 && (nw & 1u)) words[nw] = 0;
    __syncwarp();
    return nw;
}

// Receiver tables from the transmitted frequencies (f[] already in shared memory and synced): one word per slot:
// (slot - c) | symbol << 12 | (f - 1) << 20.  Returns false (in every thread) if the table does not sum to 4096.
// The owner of a slot is the last symbol that occurs and starts at or below it.  Every symbol that occurs marks the
// slot it starts at with its number + 1; a warp then carries the largest mark forward over its slots, 128 at a
// time.  (A search per thread and a walk over its 16 slots took three times the instructions, most of them diverged.)
//   base[s] = symbol << 12 | (f - 1) << 20, less c, so that a slot's word is base[owner] + slot
template <int T>
__device__ __forceinline__ bool decoder_tables(const uint16_t* f, uint16_t* c, uint32_t* base, uint32_t* tab, uint32_t* flag,
                                               uint32_t tid) {
    const uint32_t lane = tid & 31u, warp = tid >> 5;
    uint4* const tab4 = reinterpret_cast<uint4*>(tab);
#pragma unroll
    for (int i = 0; i < (int)(kProbScale / 4) / T; ++i) tab4[tid + i * T] = make_uint4(0u, 0u, 0u, 0u);
    if (tid < 32) {
        uint32_t local[8], total;
        const uint32_t first = warp_prefix256(f, tid, local, total);
#pragma unroll
        for (int i = 0; i < 8; ++i) c[8 * tid + i] = (uint16_t)min(first + local[i], kProbScale);
        if (tid == 0) *flag = total == kProbScale ? 1u : 0u;
    }
    __syncthreads();
    if (*flag == 0) return false;
    if (tid < 256u) {
        const uint32_t start = c[tid];
        base[tid] = (tid << 12 | ((uint32_t)f[tid] - 1u) << 20) - start;
        if (f[tid]) tab[start] = tid + 1u;  // f >= 1: the start is a slot, and no other symbol's start
    }
    // the owner of the slot in front of the warp's first one (mark 0: there is none)
    constexpr uint32_t kSlots = kProbScale * 32u / (uint32_t)T;  // slots of a warp
    const uint32_t slot0 = warp * kSlots;
    uint32_t carry = 0;
#pragma unroll
    for (uint32_t s = lane; s < 256u; s += 32u)
        if (f[s] && c[s] < slot0) carry = s + 1u;
    carry = __reduce_max_sync(0xffffffffu, carry);
    __syncthreads();
#pragma unroll
    for (uint32_t r = 0; r < kSlots / 128u; ++r) {
        const uint32_t slot = slot0 + 128u * r + 4u * lane;
        uint4 v = tab4[slot >> 2];
        v.y = max(v.x, v.y);
        v.z = max(v.y, v.z);
        v.w = max(v.z, v.w);
        uint32_t incl = v.w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) incl = max(incl, __shfl_up_sync(0xffffffffu, incl, o));
        uint32_t before = __shfl_up_sync(0xffffffffu, incl, 1);
        before = max(lane ? before : 0u, carry);
        carry = max(carry, __shfl_sync(0xffffffffu, incl, 31));
        // (the sum is 4096, so every slot has an owner: slot 0 is the first occurring symbol's start)
        v.x = base[max(v.x, before) - 1u] + slot;
        v.y = base[max(v.y, before) - 1u] + slot + 1u;
        v.z = base[max(v.z, before) - 1u] + slot + 2u;
        v.w = base[max(v.w, before) - 1u] + slot + 3u;
        tab4[slot >> 2] = v;
    }
    __syncthreads();
    return true;
}

// One warp decodes one segment: coded (32 states + snw words, 4-byte aligned, in global memory) ->
// out[0, n).  The words are read where they lie (a step takes a handful of neighbouring words from the
// end of what is left, so the reads of a warp fall into one or two cache lines that stay in L1 for the
// next steps); without a staged copy the kernel's shared memory is the slot table, and many warps per
// SM hide the latency of a line's first touch.
// Returns false (in every lane) if the words run out, are left over, or a lane does not end in the
// start state.  (Whether the words have run out is looked at after every four steps: they take 128 words at most, so a
// damaged section makes a lane read at most 256 bytes in front of its words -- other parts of the same message.)
// (Layer as above: 0.190 ms with the check in every step and a slot's owner searched for, 0.150 like this.)
__device__ __forceinline__ bool decode_segment(const uint8_t* coded, uint32_t snw, uint32_t n, const uint32_t* tab,
                                               uint8_t* out, uint32_t lane) {
    const uint16_t* words = reinterpret_cast<const uint16_t*>(coded + 4 * 32);
    for (uint32_t i = lane * 64u; i < snw; i += 32u * 64u)  // bring the word list towards the SM, a line per lane
        asm volatile("prefetch.global.L2 [%0];" ::"l"(words + i));
    uint32_t x = reinterpret_cast<const uint32_t*>(coded)[lane];
    int32_t ptr = (int32_t)snw;
    const uint32_t below = (1u << lane) - 1u;
    uint8_t* o = out + lane;
    auto step = [&](uint8_t* dst, bool has) {  // `has`: this lane decodes a symbol in this step
        const uint32_t en = tab[x & (kProbScale - 1u)];
        const uint32_t hi = x >> kProbBits;
        const uint32_t y = (en >> 20) * hi + hi + (en & 0xFFFu);
        if (has) {
            *dst = (uint8_t)(en >> 12);
            x = y;
        }
        const bool need = has && y < kRansL;
        const uint32_t votes = __ballot_sync(0xffffffffu, need);
        ptr -= __popc(votes);
        // (a predicated load: as an if it compiled to a branch with a reconvergence point, 0.147 -> 0.142 ms per layer)
        uint32_t w;
        asm volatile("{\n\t.reg .pred p;\n\t.reg .u16 h;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u16 h, 0;\n\t@p ld.global.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}"
                     : "=r"(w)
                     : "l"(words + (ptr + (int32_t)__popc(votes & below))), "r"((uint32_t)need)
                     : "memory");
        x = need ? __byte_perm(w, x, 0x5410u) : x;
    };
    const uint32_t full = n >> 5;  // steps in which every lane has a symbol
    uint32_t t = 0;
    for (; t + 4u <= full; t += 4u) {
#pragma unroll
        for (int k = 0; k < 4; ++k) step(o + 32 * k, true);
        o += 128;
        if (ptr < 0) return false;  // the words ran out (the same in every lane)
    }
    for (; 32u * t < n; ++t) {
        step(o, 32u * t + lane < n);
        o += 32;
    }
    const bool ok = ptr == 0 && !__any_sync(0xffffffffu, x != kRansL);
    __syncwarp();
    return ok;
}

// Raw payload length Q in bytes and symbol count S of a unit from its bitmap (block-wide; `acc` in shared
// memory, zeroed and synced by the caller).  The bitmap's bits past the last block and the pad behind it
// are zero.
template <int T>
__device__ __forceinline__ uint64_t raw_payload_bytes(const uint8_t* msg, uint64_t N, int dt, uint32_t log2b,
                                                      unsigned long long* acc, uint32_t tid, uint64_t& S) {
    const uint64_t words = (bitmap_bytes(N, log2b) + 3) >> 2;  // inside the 16-byte padded bitmap
    const uint32_t* bm32 = reinterpret_cast<const uint32_t*>(msg);
    uint32_t cnt = 0;
    for (uint64_t i = tid; i < words; i += T) cnt += __popc(bm32[i]);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if ((tid & 31u) == 0 && cnt) atomicAdd(acc, (unsigned long long)cnt);
    __syncthreads();
    // every changed block carries a full block's bytes (one per exponent; fp16: five bits per exponent, rounded up
    // to whole bytes per block), a changed short last block fewer
    const uint32_t B = 1u << log2b;
    uint64_t Q = *acc * block_payload_bytes(B, dt);
    S = *acc << log2b;
    const uint32_t rem = (uint32_t)(N & (B - 1u));
    if (rem) {
        const uint64_t kb = num_blocks(N, log2b) - 1;
        if ((msg[kb >> 3] >> (kb & 7u)) & 1u) {
            Q -= block_payload_bytes(B, dt) - block_payload_bytes(rem, dt);
            S -= B - rem;
        }
    }
    return Q;
}

// Symbol count of a sender's payload of Q bytes.  bf16, fp32: a byte each.  fp16: the changed blocks lie one
// after the other, a full one taking block_payload_bytes(B) bytes, so Q and the last block's bit (a short last
// block is the only one of another size) give the count.  0 if Q is not such a sum.
__device__ __forceinline__ uint64_t symbols_of_payload(const uint8_t* msg, uint64_t N, int dt, uint32_t log2b, uint64_t Q) {
    if (dt != CIERA_FP16) return Q;
    const uint32_t B = 1u << log2b, full = (uint32_t)block_payload_bytes(B, dt);
    const uint32_t rem = (uint32_t)(N & (B - 1u));
    uint64_t tail_bytes = 0, tail_symbols = 0;
    if (rem) {
        const uint64_t kb = num_blocks(N, log2b) - 1;
        if ((msg[kb >> 3] >> (kb & 7u)) & 1u) {
            tail_bytes = block_payload_bytes(rem, dt);
            tail_symbols = rem;
        }
    }
    if (Q < tail_bytes || (Q - tail_bytes) % full != 0) return 0;
    return ((Q - tail_bytes) / full << log2b) + tail_symbols;
}

// fp16: the symbols [lo, hi) of a payload between their packed form (five bits each, a block starting on a byte
// boundary at block index x block_payload_bytes(B); all blocks before a short last one are full) and one byte
// each.  lo is a multiple of 8 and of the block size where that is smaller; hi <= symbol count.  A group of 8
// symbols is 5 bytes: one thread moves a group.  `sym` is 8-byte aligned.
__device__ __forceinline__ uint64_t packed_group_offset(uint64_t s0, uint32_t log2b) {
    const uint32_t B = 1u << log2b;
    return (s0 >> log2b) * block_payload_bytes(B, CIERA_FP16) + (uint64_t)(((uint32_t)s0 & (B - 1u)) >> 3) * 5u;
}
__device__ __forceinline__ void unpack_symbols(const uint8_t* pay, uint8_t* sym, uint32_t log2b, uint64_t lo, uint64_t hi,
                                               uint32_t tid, uint32_t threads) {
    const uint32_t group = min(1u << log2b, 8u);
    for (uint64_t s0 = lo + (uint64_t)tid * group; s0 < hi; s0 += (uint64_t)threads * group) {
        const uint32_t ns = (uint32_t)min((uint64_t)group, hi - s0), nbytes = (5u * ns + 7u) >> 3;
        const uint8_t* src = pay + packed_group_offset(s0, log2b);
        unsigned long long v = 0;
        for (uint32_t k = 0; k < nbytes; ++k) v |= (unsigned long long)src[k] << (8u * k);
        if (ns == 8u) {
            unsigned long long out = 0;
#pragma unroll
            for (uint32_t k = 0; k < 8u; ++k) out |= ((v >> (5u * k)) & 31ull) << (8u * k);
            *reinterpret_cast<unsigned long long*>(sym + s0) = out;
        } else {
            for (uint32_t k = 0; k < ns; ++k) sym[s0 + k] = (uint8_t)((v >> (5u * k)) & 31u);
        }
    }
}
__device__ __forceinline__ void pack_symbols(const uint8_t* sym, uint8_t* pay, uint32_t log2b, uint64_t lo, uint64_t hi,
                                             uint32_t tid, uint32_t threads) {
    const uint32_t group = min(1u << log2b, 8u);
    for (uint64_t s0 = lo + (uint64_t)tid * group; s0 < hi; s0 += (uint64_t)threads * group) {
        const uint32_t ns = (uint32_t)min((uint64_t)group, hi - s0), nbytes = (5u * ns + 7u) >> 3;
        unsigned long long v = 0;
        for (uint32_t k = 0; k < ns; ++k) v |= (unsigned long long)(sym[s0 + k] & 31u) << (5u * k);
        uint8_t* dst = pay + packed_group_offset(s0, log2b);
        for (uint32_t k = 0; k < nbytes; ++k) dst[k] = (uint8_t)(v >> (8u * k));
    }
}

// Exclusive scan of one value per thread over the block; `scan` holds a word per warp.  Returns
// the thread's offset; `total` gets the block's sum.  Contains barriers.
template <int T>
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* scan, uint32_t tid, uint32_t& total) {
    const uint32_t lane = tid & 31u, warp = tid >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o) incl += t;
    }
    __syncthreads();  // the previous use of scan[] is over
    if (lane == 31) scan[warp] = incl;
    __syncthreads();
    uint32_t wbase = 0;
    total = 0;
    for (int w = 0; w < T / 32; ++w) {
        if (w < (int)warp) wbase += scan[w];
        total += scan[w];
    }
    return wbase + incl - v;
}

// ------------------------------------------------------------------------------------------ sender
// units of up to kLongSegs segment slots: one thread block per unit, start to end

template <bool HALF, int T>  // HALF: fp16, five-bit symbols (see the head of this file); T: threads of the block
__global__ void __launch_bounds__(T, T == kEntWide ? 1 : T == kEntMiddle ? 2 : 5)
entropy_encode_kernel(const ciera_unit* __restrict__ units, const unsigned long long* __restrict__ seg_base,
                      int dt, uint32_t log2b, uint8_t* msgs, unsigned long long* wire_bytes,
                      uint8_t* scratch_slots, uint32_t* scratch_nw, uint8_t* scratch_sym) {
    __shared__ uint32_t s_hist[T / 32][256];  // the warps' private histograms, then the two small lists of step 4
    __shared__ uint16_t s_f[256];
    __shared__ uint4 s_enc[256];
    __shared__ uint32_t s_scan[T / 32];
    __shared__ unsigned long long s_total;
    pdl_wait();
    const uint32_t unit = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const ciera_unit un = units[unit];
    if (un.n_values == 0 || segments_of(un.n_values) > kLongSegs) return;
    const uint64_t payoff = payload_offset_of(un.n_values, dt, log2b);
    const uint64_t Q = wire_bytes[unit] - payoff;
    // nothing to code; or a length that no sender step reports (shorter than the fixed sections, more
    // than the payload of a unit whose every block changed, not a sum of block sizes): everything below is indexed by the
    // symbol count P, so such a unit is left alone
    if (Q == 0 || Q > payload_bytes_max(un.n_values, dt, log2b)) return;
    const uint64_t P = symbols_of_payload(msgs + un.msg_off, un.n_values, dt, log2b, Q);
    if (P == 0 || P > un.n_values) return;
    uint8_t* const pay = msgs + un.msg_off + payoff;  // 16-byte aligned
    const uint32_t nseg = (uint32_t)segments_of(P);
    constexpr uint32_t hdr = HALF ? 64u : 512u;  // = model_bytes(dt)
    const uint8_t* src = pay;  // the symbols, one per byte
    if (HALF) {
        uint8_t* sym = scratch_sym + un.cache_off;
        unpack_symbols(pay, sym, log2b, 0, P, tid, T);
        src = sym;
        __syncthreads();
    }

    // 1. histogram of the symbols (one private copy per warp), 2. the model
    for (uint32_t i = lane; i < 256; i += 32) s_hist[warp][i] = 0;
    if (tid == 0) s_total = 0;
    __syncwarp();
    histogram_add<T>(s_hist, src, 0, P, tid);
    __syncthreads();
    {
        uint32_t h = 0;
        if (tid < 256u)
            for (int w = 0; w < T / 32; ++w) h += s_hist[w][tid];
        __syncthreads();
        if (tid < 256u) s_hist[0][tid] = h;
    }
    __syncthreads();
    normalise_model(s_hist[0], P, s_f, tid);
    const bool plus = encoder_tables(s_f, s_enc, tid);

    // 3. segments: warp w codes segments w, w + T / 32, ... into the unit's slots of the scratch
    const unsigned long long slot0 = seg_base[unit];
    for (uint32_t g = warp; g < nseg; g += T / 32) {
        const uint32_t n = (uint32_t)min((uint64_t)kSegment, P - (uint64_t)g * kSegment);
        const uint8_t* const seg = src + (uint64_t)g * kSegment;
        uint8_t* const slot = scratch_slots + (slot0 + g) * kSegSlot;
        const uint32_t nw = plus ? encode_segment<true>(seg, n, s_enc, slot, lane)
                                 : encode_segment<false>(seg, n, s_enc, slot, lane);
        if (lane == 0) {
            scratch_nw[slot0 + g] = nw;
            atomicAdd(&s_total, (unsigned long long)segment_bytes(nw));
        }
    }
    __syncthreads();  // every warp is done reading the raw payload and writing its slots

    // 4. keep the raw form unless the coded one is strictly shorter; else move it into the message
    const uint64_t C = (uint64_t)hdr + 4ull * nseg + s_total;
    if (C >= Q) return;
    if (tid < hdr / 2u) reinterpret_cast<uint16_t*>(pay)[tid] = s_f[tid];
    uint32_t* dir = reinterpret_cast<uint32_t*>(pay + hdr);
    uint8_t* data = pay + hdr + 4ull * nseg;
    // nseg <= kLongSegs <= T: one round
    const uint32_t nw = tid < nseg ? scratch_nw[slot0 + tid] : 0u;
    const uint32_t size = tid < nseg ? segment_bytes(nw) : 0u;
    if (tid < nseg) dir[tid] = nw;
    uint32_t total;
    uint32_t* s_off = &s_hist[1][0];
    uint32_t* s_size = &s_hist[2][0];
    const uint32_t at = block_scan<T>(size, s_scan, tid, total);
    if (tid < kLongSegs) {
        s_off[tid] = at;
        s_size[tid] = size;
    }
    __syncthreads();
    for (uint32_t k = warp; k < nseg; k += T / 32) {
        const uint32_t* from = reinterpret_cast<const uint32_t*>(scratch_slots + (slot0 + k) * kSegSlot);
        uint32_t* to = reinterpret_cast<uint32_t*>(data + s_off[k]);
        for (uint32_t i = lane; i < (s_size[k] >> 2); i += 32) to[i] = from[i];
    }
    if (tid == 0) wire_bytes[unit] = payoff + C;
}

// longer units: grids over chunks of kLongSegs segments.  A chunk record = {unit, first segment of
// the chunk inside the unit, index of the unit among the long ones, 0}.  Where the chunks are too few to fill the GPU a
// chunk is the work of several thread blocks (gridDim.y of them, a power of two), down to a segment per warp: 12 units of
// 2 097 152 values, sender's / receiver's stage 137 / 205 us with a block to a chunk, 40 / 38 like this.  Per long unit the scratch
// holds a record of 2048 bytes: 256 x u32 counts, 256 x u16 frequencies, then the words below.
constexpr uint32_t kLongRec = 2048;
// this block's segments of its chunk: first one inside the unit, and how many
__device__ __forceinline__ uint32_t part_segments() { return kLongSegs / gridDim.y; }
__device__ __forceinline__ uint32_t part_first(const uint4& chunk) { return chunk.y + blockIdx.y * part_segments(); }
struct LongState {            // at byte 1536 of a long unit's record
    unsigned long long total;   // sender: bytes of all coded segments
    unsigned long long P;       // receiver: symbols of the raw payload
    uint32_t coded;             // 1: the coded form is (sender) / was (receiver) chosen
    uint32_t bad;               // receiver: a segment did not decode
    uint32_t nseg;              // segments of the symbols
    uint32_t pad;
    unsigned long long Q;       // receiver: raw payload length in bytes (P = its symbols)
};
__device__ __forceinline__ uint32_t* long_hist(uint8_t* recs, uint32_t li) { return reinterpret_cast<uint32_t*>(recs + (size_t)li * kLongRec); }
__device__ __forceinline__ uint16_t* long_model(uint8_t* recs, uint32_t li) { return reinterpret_cast<uint16_t*>(recs + (size_t)li * kLongRec + 1024); }
__device__ __forceinline__ LongState* long_state(uint8_t* recs, uint32_t li) { return reinterpret_cast<LongState*>(recs + (size_t)li * kLongRec + 1536); }

// Symbol count of a unit's payload on the sender (0: nothing to code); Q gets the payload's length in bytes.
// A reported length that no sender step can have produced -- shorter than the fixed sections, a payload
// longer than that of a unit whose every block changed, not a sum of block sizes, e.g. the stale word of a unit that an aborted
// encode never finished -- also gives 0: the histogram, the segments and the scratch slots are all indexed
// by the symbol count, so it must stay inside the unit's slot (a value has one exponent, and plans are
// limited to units whose block counts fit 32 bits).
__device__ __forceinline__ uint64_t sender_payload(const ciera_unit& un, int dt, uint32_t log2b, const uint8_t* msgs,
                                                   const unsigned long long* wire_bytes, uint32_t unit, uint64_t& payoff,
                                                   uint64_t& Q) {
    payoff = payload_offset_of(un.n_values, dt, log2b);
    Q = wire_bytes[unit] - payoff;
    if (Q == 0 || Q > payload_bytes_max(un.n_values, dt, log2b) || Q >= (1ull << 32)) return 0;
    const uint64_t P = symbols_of_payload(msgs + un.msg_off, un.n_values, dt, log2b, Q);
    return (P <= un.n_values && P < (1ull << 32)) ? P : 0;
}
// where a unit's symbols lie, one per byte: in the message, or (fp16) unpacked in the scratch
__device__ __forceinline__ const uint8_t* sender_symbols(const ciera_unit& un, int dt, const uint8_t* msgs, uint64_t payoff,
                                                         const uint8_t* scratch_sym) {
    return dt == CIERA_FP16 ? scratch_sym + un.cache_off : msgs + un.msg_off + payoff;
}

// fp16 only: the long units' payloads unpacked into the scratch, a chunk per thread block
__global__ void __launch_bounds__(kEntThreads)
entropy_long_unpack_kernel(const ciera_unit* __restrict__ units, const uint4* __restrict__ chunks, int dt, uint32_t log2b,
                           const uint8_t* msgs, const unsigned long long* wire_bytes, uint8_t* scratch_sym) {
    pdl_wait();
    const uint4 ch = chunks[blockIdx.x];
    const ciera_unit un = units[ch.x];
    uint64_t payoff, Q;
    const uint64_t P = sender_payload(un, dt, log2b, msgs, wire_bytes, ch.x, payoff, Q);
    const uint64_t lo = (uint64_t)part_first(ch) * kSegment;
    if (lo >= P) return;
    const uint64_t hi = min(P, lo + (uint64_t)part_segments() * kSegment);
    unpack_symbols(msgs + un.msg_off + payoff, scratch_sym + un.cache_off, log2b, lo, hi, threadIdx.x, kEntThreads);
}

__global__ void __launch_bounds__(kEntThreads)
entropy_long_hist_kernel(const ciera_unit* __restrict__ units, const uint4* __restrict__ chunks, int dt, uint32_t log2b,
                         const uint8_t* msgs, const unsigned long long* wire_bytes, uint8_t* recs,
                         const uint8_t* scratch_sym) {
    __shared__ uint32_t s_hist[kEntWarps][256];
    pdl_wait();
    const uint4 ch = chunks[blockIdx.x];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const ciera_unit un = units[ch.x];
    uint64_t payoff, Q;
    const uint64_t P = sender_payload(un, dt, log2b, msgs, wire_bytes, ch.x, payoff, Q);
    const uint64_t lo = (uint64_t)part_first(ch) * kSegment;
    if (lo >= P) return;
    const uint64_t hi = min(P, lo + (uint64_t)part_segments() * kSegment);
    for (uint32_t i = lane; i < 256; i += 32) s_hist[warp][i] = 0;
    __syncwarp();
    histogram_add<kEntThreads>(s_hist, sender_symbols(un, dt, msgs, payoff, scratch_sym), lo, hi, tid);
    __syncthreads();
    uint32_t h = 0;
    for (int w = 0; w < kEntWarps; ++w) h += s_hist[w][tid];
    if (h) atomicAdd(long_hist(recs, ch.z) + tid, h);
}

__global__ void __launch_bounds__(kEntThreads)
entropy_long_model_kernel(const ciera_unit* __restrict__ units, const uint32_t* __restrict__ long_units, int dt,
                          uint32_t log2b, const uint8_t* msgs, const unsigned long long* wire_bytes, uint8_t* recs) {
    __shared__ uint32_t s_h[256];
    __shared__ uint16_t s_f[256];
    pdl_wait();
    const uint32_t li = blockIdx.x, tid = threadIdx.x, unit = long_units[li];
    uint64_t payoff, Q;
    const uint64_t P = sender_payload(units[unit], dt, log2b, msgs, wire_bytes, unit, payoff, Q);
    if (tid == 0) {
        LongState* st = long_state(recs, li);
        st->total = 0;
        st->coded = 0;
        st->bad = 0;
    }
    if (P == 0) return;
    s_h[tid] = long_hist(recs, li)[tid];
    __syncthreads();
    normalise_model(s_h, P, s_f, tid);
    long_model(recs, li)[tid] = s_f[tid];
}

template <bool HALF>  // HALF: fp16, five-bit symbols (see the head of this file)
__global__ void __launch_bounds__(kEntThreads)
entropy_long_encode_kernel(const ciera_unit* __restrict__ units, const unsigned long long* __restrict__ seg_base,
                           const uint4* __restrict__ chunks, int dt, uint32_t log2b, const uint8_t* msgs,
                           const unsigned long long* wire_bytes, uint8_t* recs, uint8_t* scratch_slots,
                           uint32_t* scratch_nw, const uint8_t* scratch_sym) {
    __shared__ uint16_t s_f[256];
    __shared__ uint4 s_enc[256];
    __shared__ unsigned long long s_total;
    pdl_wait();
    const uint4 ch = chunks[blockIdx.x];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const ciera_unit un = units[ch.x];
    uint64_t payoff, Q;
    const uint64_t P = sender_payload(un, dt, log2b, msgs, wire_bytes, ch.x, payoff, Q);
    if ((uint64_t)part_first(ch) * kSegment >= P) return;
    const uint32_t nseg = (uint32_t)segments_of(P);
    const uint32_t g_end = min(nseg, part_first(ch) + part_segments());
    s_f[tid] = long_model(recs, ch.z)[tid];
    if (tid == 0) s_total = 0;
    __syncthreads();
    const bool plus = encoder_tables(s_f, s_enc, tid);
    const uint8_t* pay = HALF ? scratch_sym + un.cache_off : msgs + un.msg_off + payoff;  // the symbols
    const unsigned long long slot0 = seg_base[ch.x];
    for (uint32_t g = part_first(ch) + warp; g < g_end; g += kEntWarps) {
        const uint32_t n = (uint32_t)min((uint64_t)kSegment, P - (uint64_t)g * kSegment);
        const uint8_t* const seg = pay + (uint64_t)g * kSegment;
        uint8_t* const slot = scratch_slots + (slot0 + g) * kSegSlot;
        const uint32_t nw = plus ? encode_segment<true>(seg, n, s_enc, slot, lane)
                                 : encode_segment<false>(seg, n, s_enc, slot, lane);
        if (lane == 0) {
            scratch_nw[slot0 + g] = nw;
            atomicAdd(&s_total, (unsigned long long)segment_bytes(nw));
        }
    }
    __syncthreads();
    if (tid == 0) atomicAdd(&long_state(recs, ch.z)->total, s_total);
}

// decides raw or coded for a long unit; coded: table and word counts into the message, the byte
// offset of every segment into the scratch
__global__ void __launch_bounds__(kEntThreads)
entropy_long_layout_kernel(const ciera_unit* __restrict__ units, const unsigned long long* __restrict__ seg_base,
                           const uint32_t* __restrict__ long_units, int dt, uint32_t log2b, uint8_t* msgs,
                           unsigned long long* wire_bytes, uint8_t* recs, const uint32_t* scratch_nw,
                           uint32_t* scratch_off) {
    __shared__ uint32_t s_scan[kEntWarps];
    pdl_wait();
    const uint32_t li = blockIdx.x, tid = threadIdx.x, unit = long_units[li];
    const ciera_unit un = units[unit];
    uint64_t payoff, Q;
    const uint64_t P = sender_payload(un, dt, log2b, msgs, wire_bytes, unit, payoff, Q);
    if (P == 0) return;
    const uint32_t nseg = (uint32_t)segments_of(P);
    const uint32_t hdr = model_bytes(dt);
    LongState* st = long_state(recs, li);
    const uint64_t C = (uint64_t)hdr + 4ull * nseg + st->total;
    if (C >= Q) return;
    uint8_t* pay = msgs + un.msg_off + payoff;
    if (tid < hdr / 2u) reinterpret_cast<uint16_t*>(pay)[tid] = long_model(recs, li)[tid];
    uint32_t* dir = reinterpret_cast<uint32_t*>(pay + hdr);
    const unsigned long long slot0 = seg_base[unit];
    uint32_t carry = 0;  // C < Q < 2^32: offsets fit
    for (uint32_t g0 = 0; g0 < nseg; g0 += kEntThreads) {
        const uint32_t g = g0 + tid;
        const uint32_t nw = g < nseg ? scratch_nw[slot0 + g] : 0u;
        if (g < nseg) dir[g] = nw;
        uint32_t total;
        const uint32_t off = block_scan<kEntThreads>(g < nseg ? segment_bytes(nw) : 0u, s_scan, tid, total);
        if (g < nseg) scratch_off[slot0 + g] = carry + off;
        carry += total;
    }
    if (tid == 0) {
        st->coded = 1;
        st->nseg = nseg;
        wire_bytes[unit] = payoff + C;
    }
}

__global__ void __launch_bounds__(kEntThreads)
entropy_long_copy_kernel(const ciera_unit* __restrict__ units, const unsigned long long* __restrict__ seg_base,
                         const uint4* __restrict__ chunks, int dt, uint32_t log2b, uint8_t* msgs, uint8_t* recs,
                         const uint8_t* scratch_slots, const uint32_t* scratch_nw, const uint32_t* scratch_off) {
    pdl_wait();
    const uint4 ch = chunks[blockIdx.x];
    const LongState* st = long_state(recs, ch.z);
    if (st->coded == 0) return;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const ciera_unit un = units[ch.x];
    const uint32_t nseg = st->nseg;
    uint8_t* data = msgs + un.msg_off + payload_offset_of(un.n_values, dt, log2b) + model_bytes(dt) + 4ull * nseg;
    const unsigned long long slot0 = seg_base[ch.x];
    const uint32_t g_end = min(nseg, part_first(ch) + part_segments());
    for (uint32_t g = part_first(ch) + warp; g < g_end; g += kEntWarps) {
        const uint32_t* from = reinterpret_cast<const uint32_t*>(scratch_slots + (slot0 + g) * kSegSlot);
        uint32_t* to = reinterpret_cast<uint32_t*>(data + scratch_off[slot0 + g]);
        const uint32_t words4 = segment_bytes(scratch_nw[slot0 + g]) >> 2;
        for (uint32_t i = lane; i < words4; i += 32) to[i] = from[i];
    }
}

// ---------------------------------------------------------------------------------------- receiver
// units of up to kLongSegs segment slots: one thread block per unit, start to end

struct DecodeShared {
    uint32_t tab[kProbScale];      // slot -> (slot - c) | symbol << 12 | (f - 1) << 20
    uint16_t f[256], c[256];
    uint32_t base[256];            // per symbol: see decoder_tables
    uint32_t off[kLongSegs];       // per segment: byte offset in the data part
    uint32_t nw[kLongSegs];        //              word count
    uint32_t scan[kEntWide / 32];
    unsigned long long changed;    // set bits of the unit's bitmap
    uint32_t flag, bad;
};

__device__ __forceinline__ void raise_corrupt(int32_t* status) {
    if (status) atomicCAS(status, 0, (int32_t)CIERA_ERR_CORRUPT);
}

// HALF: fp16, five-bit symbols (see the head of this file); T: threads of the block; BLOCKS: blocks per SM it is built for
// (8 blocks leave 32 registers: 0.142 ms per OLMoE-shaped layer against 0.166 with 5; but where the units do not fill
// more than 5, the 48 registers shorten the chain: 512 units 55 us against 70, 192 units 48 against 57)
template <bool HALF, int T, int BLOCKS>
__global__ void __launch_bounds__(T, BLOCKS)
entropy_decode_kernel(const ciera_unit* __restrict__ units, int dt, uint32_t log2b, uint8_t* msgs,
                      unsigned long long* wire_bytes, uint8_t* scratch_raw, int32_t* status) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    DecodeShared& sh = *reinterpret_cast<DecodeShared*>(smem_raw);
    pdl_wait();
    const uint32_t unit = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const ciera_unit un = units[unit];
    const uint64_t N = un.n_values;
    if (N == 0 || segments_of(N) > kLongSegs) return;
    uint8_t* const msg = msgs + un.msg_off;
    const uint64_t payoff = payload_offset_of(N, dt, log2b);
    if (tid == 0) {
        sh.changed = 0;
        sh.bad = 0;
    }
    __syncthreads();
    uint64_t P;  // symbols; Q = bytes of the raw payload
    const uint64_t Q = raw_payload_bytes<T>(msg, N, dt, log2b, &sh.changed, tid, P);
    const uint64_t wire = wire_bytes[unit];
    if (Q == 0 || wire == payoff + Q) return;  // nothing travelled, or the raw form did
    const uint64_t C = wire - payoff;
    const uint32_t nseg = (uint32_t)segments_of(P);
    constexpr uint32_t hdr = HALF ? 64u : 512u;  // = model_bytes(dt)
    uint8_t* const pay = msg + payoff;
    if (wire < payoff || C >= Q || C < (uint64_t)hdr + 4ull * nseg) {
        if (tid == 0) raise_corrupt(status);
        return;
    }
    if (tid < 256u) sh.f[tid] = tid < hdr / 2u ? reinterpret_cast<const uint16_t*>(pay)[tid] : (uint16_t)0;
    __syncthreads();
    if (!decoder_tables<T>(sh.f, sh.c, sh.base, sh.tab, &sh.flag, tid)) {
        if (tid == 0) raise_corrupt(status);
        return;
    }
    // where the segments lie (nseg <= kLongSegs <= T: one round)
    const uint32_t* dir = reinterpret_cast<const uint32_t*>(pay + hdr);
    const uint8_t* data = pay + hdr + 4ull * nseg;
    const uint64_t data_bytes = C - hdr - 4ull * nseg;
    const uint32_t nw = tid < nseg ? dir[tid] : 0u;
    if (nw > kSegWordsMax) sh.bad = 1;
    uint32_t total;
    const uint32_t at = block_scan<T>(tid < nseg ? segment_bytes(min(nw, kSegWordsMax)) : 0u, sh.scan, tid, total);
    if (tid < kLongSegs) {
        sh.off[tid] = at;
        sh.nw[tid] = min(nw, kSegWordsMax);
    }
    __syncthreads();
    if (sh.bad || total != data_bytes) {
        if (tid == 0) raise_corrupt(status);
        return;
    }
    uint8_t* raw = scratch_raw + un.cache_off;  // the unit's stretch of the scratch (16-byte aligned)
    for (uint32_t g = warp; g < nseg; g += T / 32) {
        const uint32_t n = (uint32_t)min((uint64_t)kSegment, P - (uint64_t)g * kSegment);
        if (!decode_segment(data + sh.off[g], sh.nw[g], n, sh.tab, raw + (uint64_t)g * kSegment, lane))
            sh.bad = 1;
    }
    __syncthreads();
    if (sh.bad) {
        if (tid == 0) raise_corrupt(status);
        return;
    }
    // the raw payload goes back into the message, which then is what the sender step had written
    if (HALF) {
        pack_symbols(raw, pay, log2b, 0, P, tid, T);
    } else {
        for (uint64_t i = (uint64_t)tid * 16; i < P; i += (uint64_t)T * 16) {
            if (i + 16 <= P) {
                *reinterpret_cast<uint4*>(pay + i) = *reinterpret_cast<const uint4*>(raw + i);
            } else {
                for (uint64_t k = i; k < P; ++k) pay[k] = raw[k];
            }
        }
    }
    if (tid == 0) wire_bytes[unit] = payoff + Q;
}

// longer units: layout (one block per unit), segments and restore (grids over chunks)
__global__ void __launch_bounds__(kEntThreads)
entropy_long_parse_kernel(const ciera_unit* __restrict__ units, const unsigned long long* __restrict__ seg_base,
                          const uint32_t* __restrict__ long_units, int dt, uint32_t log2b, const uint8_t* msgs,
                          const unsigned long long* wire_bytes, uint8_t* recs, uint32_t* scratch_off, uint32_t* scratch_nw,
                          int32_t* status) {
    __shared__ uint32_t s_scan[kEntWarps];
    __shared__ unsigned long long s_changed;
    __shared__ uint32_t s_bad;
    pdl_wait();
    const uint32_t li = blockIdx.x, tid = threadIdx.x, unit = long_units[li];
    const ciera_unit un = units[unit];
    const uint64_t N = un.n_values;
    LongState* st = long_state(recs, li);
    if (tid == 0) {
        st->coded = 0;
        st->bad = 0;
        s_changed = 0;
        s_bad = 0;
    }
    __syncthreads();
    const uint8_t* msg = msgs + un.msg_off;
    const uint64_t payoff = payload_offset_of(N, dt, log2b);
    uint64_t P;  // symbols; Q = bytes of the raw payload
    const uint64_t Q = raw_payload_bytes<kEntThreads>(msg, N, dt, log2b, &s_changed, tid, P);
    const uint64_t wire = wire_bytes[unit];
    if (Q == 0 || wire == payoff + Q) return;
    const uint64_t C = wire - payoff;
    const uint64_t nseg64 = segments_of(P);
    const uint32_t hdr = model_bytes(dt);
    if (wire < payoff || C >= Q || P >= (1ull << 32) || C < (uint64_t)hdr + 4ull * nseg64) {
        if (tid == 0) raise_corrupt(status);
        return;
    }
    const uint32_t nseg = (uint32_t)nseg64;
    const uint8_t* pay = msg + payoff;
    const uint32_t* dir = reinterpret_cast<const uint32_t*>(pay + hdr);
    const uint64_t data_bytes = C - hdr - 4ull * nseg;
    const unsigned long long slot0 = seg_base[unit];
    uint64_t carry = 0;
    for (uint32_t g0 = 0; g0 < nseg; g0 += kEntThreads) {
        const uint32_t g = g0 + tid;
        const uint32_t nw = g < nseg ? dir[g] : 0u;
        if (nw > kSegWordsMax) s_bad = 1;
        uint32_t total;
        const uint32_t off = block_scan<kEntThreads>(g < nseg ? segment_bytes(min(nw, kSegWordsMax)) : 0u, s_scan, tid, total);
        if (g < nseg) {
            scratch_off[slot0 + g] = (uint32_t)(carry + off);
            scratch_nw[slot0 + g] = min(nw, kSegWordsMax);
        }
        carry += total;
    }
    __syncthreads();
    if (s_bad || carry != data_bytes) {
        if (tid == 0) raise_corrupt(status);
        return;
    }
    if (tid == 0) {
        st->P = P;
        st->Q = Q;
        st->nseg = nseg;
        st->coded = 1;
    }
}

template <bool HALF>  // HALF: fp16, five-bit symbols (see the head of this file)
__global__ void __launch_bounds__(kEntThreads)
entropy_long_decode_kernel(const ciera_unit* __restrict__ units, const unsigned long long* __restrict__ seg_base,
                           const uint4* __restrict__ chunks, int dt, uint32_t log2b, const uint8_t* msgs,
                           uint8_t* recs, const uint32_t* scratch_off, const uint32_t* scratch_nw, uint8_t* scratch_raw,
                           int32_t* status) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    DecodeShared& sh = *reinterpret_cast<DecodeShared*>(smem_raw);
    pdl_wait();
    const uint4 ch = chunks[blockIdx.x];
    LongState* st = long_state(recs, ch.z);
    if (st->coded == 0 || part_first(ch) >= st->nseg) return;
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const ciera_unit un = units[ch.x];
    const uint64_t P = st->P;
    const uint32_t nseg = st->nseg;
    const uint8_t* pay = msgs + un.msg_off + payload_offset_of(un.n_values, dt, log2b);
    constexpr uint32_t hdr = HALF ? 64u : 512u;  // = model_bytes(dt)
    sh.f[tid] = tid < hdr / 2u ? reinterpret_cast<const uint16_t*>(pay)[tid] : (uint16_t)0;
    if (tid == 0) sh.bad = 0;
    __syncthreads();
    if (!decoder_tables<kEntThreads>(sh.f, sh.c, sh.base, sh.tab, &sh.flag, tid)) {
        if (tid == 0) {
            st->bad = 1;
            raise_corrupt(status);
        }
        return;
    }
    const uint8_t* data = pay + hdr + 4ull * nseg;
    uint8_t* raw = scratch_raw + un.cache_off;
    const unsigned long long slot0 = seg_base[ch.x];
    const uint32_t g_end = min(nseg, part_first(ch) + part_segments());
    for (uint32_t g = part_first(ch) + warp; g < g_end; g += kEntWarps) {
        const uint32_t n = (uint32_t)min((uint64_t)kSegment, P - (uint64_t)g * kSegment);
        if (!decode_segment(data + scratch_off[slot0 + g], scratch_nw[slot0 + g], n, sh.tab,
                            raw + (uint64_t)g * kSegment, lane))
            sh.bad = 1;
    }
    __syncthreads();
    if (tid == 0 && sh.bad) {
        st->bad = 1;
        raise_corrupt(status);
    }
}

__global__ void __launch_bounds__(kEntThreads)
entropy_long_restore_kernel(const ciera_unit* __restrict__ units, const uint4* __restrict__ chunks, int dt,
                            uint32_t log2b, uint8_t* msgs, unsigned long long* wire_bytes, const uint8_t* recs_c,
                            const uint8_t* scratch_raw) {
    pdl_wait();
    const uint4 ch = chunks[blockIdx.x];
    const LongState* st = long_state(const_cast<uint8_t*>(recs_c), ch.z);
    if (st->coded == 0 || st->bad != 0) return;  // raw as received, or damaged: left as it is
    const uint32_t tid = threadIdx.x;
    const ciera_unit un = units[ch.x];
    const uint64_t P = st->P;
    const uint64_t lo = (uint64_t)part_first(ch) * kSegment;
    if (lo >= P) return;
    const uint64_t hi = min(P, lo + (uint64_t)part_segments() * kSegment);
    const uint64_t payoff = payload_offset_of(un.n_values, dt, log2b);
    uint8_t* pay = msgs + un.msg_off + payoff;
    const uint8_t* raw = scratch_raw + un.cache_off;
    if (dt == CIERA_FP16) {
        pack_symbols(raw, pay, log2b, lo, hi, tid, kEntThreads);
    } else {
        for (uint64_t i = lo + (uint64_t)tid * 16; i < hi; i += (uint64_t)kEntThreads * 16) {
            if (i + 16 <= hi) {
                *reinterpret_cast<uint4*>(pay + i) = *reinterpret_cast<const uint4*>(raw + i);
            } else {
                for (uint64_t k = i; k < hi; ++k) pay[k] = raw[k];
            }
        }
    }
    if (lo == 0 && tid == 0) wire_bytes[ch.x] = payoff + st->Q;
}

}  // namespace ciera

using namespace ciera;

static bool misaligned16(const void* p) { return ((uintptr_t)p & 15u) != 0; }
static size_t up16(size_t x) { return (x + 15) / 16 * 16; }

// Scratch: [word count per segment slot][byte offset per segment slot][a record per long unit]
// [body: the segment slots (sender) or the decoded symbols at the units' cache offsets (receiver)]
// [fp16 sender: the unpacked symbols at the units' cache offsets]
struct ScratchLayout {
    size_t nw, off, recs, body, sym, total;
};
static ScratchLayout scratch_layout(const ciera_plan* p) {
    ScratchLayout L;
    L.nw = 0;
    L.off = L.nw + up16((size_t)p->total_segments * sizeof(uint32_t));
    L.recs = L.off + up16((size_t)p->total_segments * sizeof(uint32_t));
    L.body = L.recs + (size_t)p->ent_long_units.size() * kLongRec;
    const size_t enc = (size_t)p->total_segments * kSegSlot, dec = (size_t)p->cache_extent;
    L.sym = L.body + up16(enc > dec ? enc : dec);
    L.total = L.sym + (p->dtype == CIERA_FP16 ? dec : 0) + 16;
    return L;
}

extern "C" size_t ciera_plan_entropy_scratch_bytes(const ciera_plan* p) { return p ? scratch_layout(p).total : 0; }

static int check_entropy_args(const ciera_plan* p, const void* messages_dev, const void* wire_bytes_dev,
                              const void* scratch_dev) {
    if (!p) return CIERA_ERR_INVALID_ARG;
    if (!p->tiles.empty() && !p->tiles_dev) return CIERA_ERR_NOT_BOUND;
    if (p->tiles.empty()) return CIERA_OK;
    if (!messages_dev || !wire_bytes_dev || !scratch_dev) return CIERA_ERR_INVALID_ARG;
    if (misaligned16(messages_dev) || misaligned16(scratch_dev) || ((uintptr_t)wire_bytes_dev & 7u))
        return CIERA_ERR_MISALIGNED;
    return CIERA_OK;
}

// SMs of the current device, and the dynamic shared memory of the receiver's kernels set up once per device
static int entropy_device(int* sms_out) {
    static std::atomic<int> cached[64];  // (zero-initialised; any host thread may be the first to fill an entry)
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda_error(e);
    if (dev < 0 || dev >= 64) return CIERA_ERR_UNSUPPORTED;
    if (!cached[dev].load(std::memory_order_acquire)) {
        for (const void* k : {(const void*)entropy_decode_kernel<false, kEntThreads, 5>, (const void*)entropy_decode_kernel<true, kEntThreads, 5>,
                              (const void*)entropy_decode_kernel<false, kEntThreads, 8>, (const void*)entropy_decode_kernel<true, kEntThreads, 8>,
                              (const void*)entropy_decode_kernel<false, kEntMiddle, 2>, (const void*)entropy_decode_kernel<true, kEntMiddle, 2>, (const void*)entropy_decode_kernel<false, kEntWide, 1>, (const void*)entropy_decode_kernel<true, kEntWide, 1>,
                              (const void*)entropy_long_decode_kernel<false>, (const void*)entropy_long_decode_kernel<true>}) {
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DecodeShared));
            if (e != cudaSuccess) return record_cuda_error(e);
        }
        int sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return record_cuda_error(e);
        if (sms < 1) return CIERA_ERR_UNSUPPORTED;
        cached[dev].store(sms, std::memory_order_release);
    }
    *sms_out = cached[dev].load(std::memory_order_acquire);
    return CIERA_OK;
}
// threads of the blocks that code a unit each
static int unit_threads(uint32_t units, int sms) {
    return units <= (uint32_t)sms ? kEntWide : units <= 2u * (uint32_t)sms ? kEntMiddle : kEntThreads;
}
// thread blocks to a chunk of kLongSegs segments: enough for five on every SM, at least a segment for each of their warps
static uint32_t chunk_parts(uint32_t chunks, int sms) {
    uint32_t parts = 1;
    while (parts < kLongSegs / kEntWarps && chunks * parts < 5u * (uint32_t)sms) parts *= 2;
    return parts;
}

extern "C" int ciera_entropy_encode(const ciera_plan* p, void* messages_dev, uint64_t* wire_bytes_dev, void* scratch_dev,
                                    void* stream) {
    int rc = check_entropy_args(p, messages_dev, wire_bytes_dev, scratch_dev);
    if (rc || p->tiles.empty()) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    const ScratchLayout L = scratch_layout(p);
    uint8_t* base = (uint8_t*)scratch_dev;
    uint32_t* nw = (uint32_t*)(base + L.nw);
    uint32_t* off = (uint32_t*)(base + L.off);
    uint8_t* recs = base + L.recs;
    uint8_t* slots = base + L.body;
    uint8_t* sym = base + L.sym;
    const int dt = p->dtype;
    uint8_t* msgs = (uint8_t*)messages_dev;
    unsigned long long* wire = (unsigned long long*)wire_bytes_dev;
    const uint32_t n_long = (uint32_t)p->ent_long_units.size(), n_chunks = (uint32_t)p->ent_chunks.size();
    int sms = 0;
    if ((rc = entropy_device(&sms))) return rc;
    cudaError_t e = cudaSuccess;
    if (n_long < p->n_units) {
        const int threads = unit_threads(p->n_units - n_long, sms);
        auto pick = [&](auto half) {
            constexpr bool kHalf = decltype(half)::value;
            return threads == kEntWide     ? entropy_encode_kernel<kHalf, kEntWide>
                   : threads == kEntMiddle ? entropy_encode_kernel<kHalf, kEntMiddle>
                                           : entropy_encode_kernel<kHalf, kEntThreads>;
        };
        e = launch_when(threads == kEntWide, dt == CIERA_FP16 ? pick(std::true_type{}) : pick(std::false_type{}), dim3(p->n_units),
                        threads, 0, s, p->units_dev, p->seg_base_dev, dt, p->log2b, msgs, wire, slots, nw, sym);
        if (e != cudaSuccess) return record_cuda_error(e);
        count_launch();
    }
    if (n_long) {
        const dim3 parts(n_chunks, chunk_parts(n_chunks, sms));
        auto launch = [&](auto* k, dim3 grid, auto... args) {
            if (e == cudaSuccess) e = launch_after(k, grid, kEntThreads, 0, s, args...);
            if (e == cudaSuccess) count_launch();
        };
        e = cudaMemsetAsync(recs, 0, (size_t)n_long * kLongRec, s);  // the counts start at zero
        if (dt == CIERA_FP16) launch(entropy_long_unpack_kernel, parts, p->units_dev, p->ent_chunks_dev, dt, p->log2b, msgs, wire, sym);
        launch(entropy_long_hist_kernel, parts, p->units_dev, p->ent_chunks_dev, dt, p->log2b, msgs, wire, recs, sym);
        launch(entropy_long_model_kernel, dim3(n_long), p->units_dev, p->ent_long_units_dev, dt, p->log2b, msgs, wire, recs);
        launch(dt == CIERA_FP16 ? entropy_long_encode_kernel<true> : entropy_long_encode_kernel<false>, parts, p->units_dev,
               p->seg_base_dev, p->ent_chunks_dev, dt, p->log2b, msgs, wire, recs, slots, nw, sym);
        launch(entropy_long_layout_kernel, dim3(n_long), p->units_dev, p->seg_base_dev, p->ent_long_units_dev, dt, p->log2b, msgs,
               wire, recs, nw, off);
        launch(entropy_long_copy_kernel, parts, p->units_dev, p->seg_base_dev, p->ent_chunks_dev, dt, p->log2b, msgs, recs, slots,
               nw, off);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    return CIERA_OK;
}

extern "C" int ciera_entropy_decode(const ciera_plan* p, void* messages_dev, uint64_t* wire_bytes_dev, void* scratch_dev,
                                    int32_t* status_dev, void* stream) {
    int rc = check_entropy_args(p, messages_dev, wire_bytes_dev, scratch_dev);
    if (rc || p->tiles.empty()) return rc;
    int sms = 0;
    if ((rc = entropy_device(&sms))) return rc;
    cudaError_t e = cudaSuccess;
    cudaStream_t s = (cudaStream_t)stream;
    const ScratchLayout L = scratch_layout(p);
    uint8_t* base = (uint8_t*)scratch_dev;
    uint32_t* nw = (uint32_t*)(base + L.nw);
    uint32_t* off = (uint32_t*)(base + L.off);
    uint8_t* recs = base + L.recs;
    uint8_t* raw = base + L.body;
    const int dt = p->dtype;
    uint8_t* msgs = (uint8_t*)messages_dev;
    unsigned long long* wire = (unsigned long long*)wire_bytes_dev;
    const uint32_t n_long = (uint32_t)p->ent_long_units.size(), n_chunks = (uint32_t)p->ent_chunks.size();
    if (n_long < p->n_units) {
        const int threads = unit_threads(p->n_units - n_long, sms);
        const bool few = p->n_units - n_long <= 5u * (uint32_t)sms;  // (see entropy_decode_kernel)
        auto pick = [&](auto half) {
            constexpr bool kHalf = decltype(half)::value;
            return threads == kEntWide     ? entropy_decode_kernel<kHalf, kEntWide, 1>
                   : threads == kEntMiddle ? entropy_decode_kernel<kHalf, kEntMiddle, 2>
                   : few                   ? entropy_decode_kernel<kHalf, kEntThreads, 5>
                                           : entropy_decode_kernel<kHalf, kEntThreads, 8>;
        };
        e = launch_when(threads == kEntWide, dt == CIERA_FP16 ? pick(std::true_type{}) : pick(std::false_type{}), dim3(p->n_units),
                        threads, sizeof(DecodeShared), s, p->units_dev, dt, p->log2b, msgs, wire, raw, status_dev);
        if (e != cudaSuccess) return record_cuda_error(e);
        count_launch();
    }
    if (n_long) {
        const dim3 parts(n_chunks, chunk_parts(n_chunks, sms));
        auto launch = [&](auto* k, dim3 grid, size_t smem, auto... args) {
            if (e == cudaSuccess) e = launch_after(k, grid, kEntThreads, smem, s, args...);
            if (e == cudaSuccess) count_launch();
        };
        launch(entropy_long_parse_kernel, dim3(n_long), 0, p->units_dev, p->seg_base_dev, p->ent_long_units_dev, dt, p->log2b, msgs,
               wire, recs, off, nw, status_dev);
        launch(dt == CIERA_FP16 ? entropy_long_decode_kernel<true> : entropy_long_decode_kernel<false>, parts, sizeof(DecodeShared),
               p->units_dev, p->seg_base_dev, p->ent_chunks_dev, dt, p->log2b, msgs, recs, off, nw, raw, status_dev);
        launch(entropy_long_restore_kernel, parts, 0, p->units_dev, p->ent_chunks_dev, dt, p->log2b, msgs, wire, recs, raw);
        if (e != cudaSuccess) return record_cuda_error(e);
    }
    return CIERA_OK;
}
