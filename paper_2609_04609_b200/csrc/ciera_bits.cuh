// Per-thread register work on "pieces": runs of consecutive values owned by one thread.
//
// Split and merge follow the paper's Section 3.1 (a value is sign, exponent and mantissa bits;
// the exponent travels apart from sign-plus-mantissa) on the IEEE binary32 / bfloat16 layouts:
//   bf16: bit 15 sign, bits 14:7 exponent, bits 6:0 mantissa  -> sm byte  = sign<<7  | mantissa
//   fp32: bit 31 sign, bits 30:23 exponent, bits 22:0 mantissa -> sm 24bit = sign<<23 | mantissa
// Everything is done on packed 32-bit words with shifts, three-input logic and byte permutes,
// four values at a time.
//
// Thread -> value layout inside a tile of 8192 values (512 consumer threads):
//   bf16: two pieces of 8 values per thread, piece p of thread t = values [4096 p + 8 t, +8).
//         Every access of a warp is then one contiguous run: 16 B / lane on the weights,
//         8 B / lane on the byte-wide streams (exponents, sign-plus-mantissa).
//   fp32: one piece of 16 values per thread, values [16 t, +16): 64 B of weights, 16 B of
//         exponents, 48 B of sign-plus-mantissa per lane.
// With blocks of 16 values and more a piece never straddles a block, so a piece has one "my
// exponents changed" bit; the tile has 1024 (bf16) or 512 (fp32) such bits.  With smaller blocks
// a piece holds 1 to 16 whole blocks and has one bit for each.
#pragma once

#include "ciera_internal.cuh"

namespace ciera {

// ---- 8- and 16-byte accesses ---------------------------------------------------------------
__device__ __forceinline__ uint4 ld_stream16(const void* p) { return __ldcs(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ uint2 ld_stream8(const void* p) { return __ldcs(reinterpret_cast<const uint2*>(p)); }
__device__ __forceinline__ void st_stream16(void* p, uint4 v) { __stcs(reinterpret_cast<uint4*>(p), v); }
__device__ __forceinline__ void st_stream8(void* p, uint2 v) { __stcs(reinterpret_cast<uint2*>(p), v); }
__device__ __forceinline__ uint4 ld_shared16(const void* p) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
    return v;
}
__device__ __forceinline__ uint2 ld_shared8(const void* p) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"((uint32_t)__cvta_generic_to_shared(p)));
    return v;
}
__device__ __forceinline__ void st_shared16(void* p, uint4 v) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ void st_shared8(void* p, uint2 v) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"((uint32_t)__cvta_generic_to_shared(p)), "r"(v.x), "r"(v.y)
                 : "memory");
}
// memory spaces a piece is read from / written to
struct Global {
    static __device__ __forceinline__ uint4 ld16(const uint8_t* p) { return ld_stream16(p); }
    static __device__ __forceinline__ uint2 ld8(const uint8_t* p) { return ld_stream8(p); }
    static __device__ __forceinline__ void st16(uint8_t* p, uint4 v) { st_stream16(p, v); }
    static __device__ __forceinline__ void st8(uint8_t* p, uint2 v) { st_stream8(p, v); }
    static __device__ __forceinline__ uint32_t ld1(const uint8_t* p) { return __ldcs(p); }
    static __device__ __forceinline__ uint32_t ld2(const uint8_t* p) { return __ldcs(reinterpret_cast<const uint16_t*>(p)); }
    static __device__ __forceinline__ uint32_t ld4(const uint8_t* p) { return __ldcs(reinterpret_cast<const uint32_t*>(p)); }
};
struct Shared {
    static __device__ __forceinline__ uint4 ld16(const uint8_t* p) { return ld_shared16(p); }
    static __device__ __forceinline__ uint2 ld8(const uint8_t* p) { return ld_shared8(p); }
    static __device__ __forceinline__ void st16(uint8_t* p, uint4 v) { st_shared16(p, v); }
    static __device__ __forceinline__ void st8(uint8_t* p, uint2 v) { st_shared8(p, v); }
    static __device__ __forceinline__ uint32_t ld1(const uint8_t* p) {
        uint32_t v;
        asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)));
        return v;
    }
    static __device__ __forceinline__ uint32_t ld2(const uint8_t* p) {
        uint32_t v;
        asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)));
        return v;
    }
    static __device__ __forceinline__ uint32_t ld4(const uint8_t* p) {
        uint32_t v;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"((uint32_t)__cvta_generic_to_shared(p)));
        return v;
    }
};

// (x & mask) | (y & ~mask): one three-input logic operation
__device__ __forceinline__ uint32_t bitselect(uint32_t mask, uint32_t x, uint32_t y) { return (x & mask) | (y & ~mask); }

// ---- bf16 --------------------------------------------------------------------------------
// Four values a = v0 | v1 << 16, b = v2 | v3 << 16.  Gather their low bytes (e0 m6..m0) and high
// bytes (s e7..e1) with two byte permutes; then
//   sm byte  = (high & 0x80) | (low & 0x7F)            exponent byte = (high << 1) | (low >> 7)
// for all four at once (the shifts leak across byte lanes only into bits that are masked off).
__device__ __forceinline__ void bf16_split4(uint32_t a, uint32_t b, uint32_t& e, uint32_t& sm) {
    const uint32_t lo = __byte_perm(a, b, 0x6420), hi = __byte_perm(a, b, 0x7531);
    sm = bitselect(0x7F7F7F7Fu, lo, hi);
    e = bitselect(0xFEFEFEFEu, hi << 1, lo >> 7);
}
// four exponent bytes + four sm bytes -> two words of two bf16 each
__device__ __forceinline__ void bf16_merge4(uint32_t e, uint32_t s, uint32_t& a, uint32_t& b) {
    const uint32_t lo = bitselect(0x7F7F7F7Fu, s, e << 7);  // e0 m6..m0
    const uint32_t hi = bitselect(0x80808080u, s, e >> 1);  // s e7..e1
    a = __byte_perm(lo, hi, 0x5140);
    b = __byte_perm(lo, hi, 0x7362);
}

// ---- fp32 --------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t fp32_exp4(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
    uint32_t t01 = __byte_perm(w0 << 1, w1 << 1, 0x0073);  // byte0 = exp(w0), byte1 = exp(w1)
    uint32_t t23 = __byte_perm(w2 << 1, w3 << 1, 0x0073);
    return __byte_perm(t01, t23, 0x5410);
}
// sign << 23 | mantissa in bits 23:0 (bits 31:24 are don't-care for the packing below)
__device__ __forceinline__ uint32_t fp32_sm(uint32_t w) { return bitselect(0x007FFFFFu, w, w >> 8); }
// four 24-bit sm values -> three little-endian words
__device__ __forceinline__ void fp32_pack4(uint32_t s0, uint32_t s1, uint32_t s2, uint32_t s3, uint32_t& o0,
                                           uint32_t& o1, uint32_t& o2) {
    o0 = __byte_perm(s0, s1, 0x4210);
    o1 = __byte_perm(s1, s2, 0x5421);
    o2 = __byte_perm(s2, s3, 0x6542);
}
// three words -> four sm values in bits 23:0 (bits 31:24 don't-care)
__device__ __forceinline__ void fp32_unpack4(uint32_t o0, uint32_t o1, uint32_t o2, uint32_t& s0, uint32_t& s1,
                                             uint32_t& s2, uint32_t& s3) {
    s0 = o0;
    s1 = __byte_perm(o0, o1, 0x0543);
    s2 = __byte_perm(o1, o2, 0x0432);
    s3 = o2 >> 8;
}
// exponent in bits 7:0 of e (higher bits don't-care), sm in bits 23:0 of s
__device__ __forceinline__ uint32_t fp32_merge(uint32_t e, uint32_t s) {
    return bitselect(0x007FFFFFu, s, bitselect(0x7F800000u, e << 23, s << 8));
}

// ---- byte-granular access to a short run of exponent / sm bytes held in words ---------------
template <int NB>
__device__ __forceinline__ void load_bytes_partial(uint32_t* w, const uint8_t* src, int nbytes) {
#pragma unroll
    for (int i = 0; i < NB / 4; ++i) w[i] = 0;
#pragma unroll
    for (int i = 0; i < NB; ++i)
        if (i < nbytes) w[i >> 2] |= (uint32_t)src[i] << (8 * (i & 3));
}
template <int NB>
__device__ __forceinline__ void store_bytes_partial(uint8_t* dst, const uint32_t* w, int nbytes) {
#pragma unroll
    for (int i = 0; i < NB; ++i)
        if (i < nbytes) dst[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
}
template <int NH>
__device__ __forceinline__ void store_halves_partial(uint8_t* dst, const uint32_t* w, int nhalves) {
    uint16_t* const p = reinterpret_cast<uint16_t*>(dst);
#pragma unroll
    for (int i = 0; i < NH; ++i)
        if (i < nhalves) p[i] = (uint16_t)(w[i >> 1] >> (16 * (i & 1)));
}
__device__ __forceinline__ void load_16_bytes(const uint8_t* src, uint32_t* w) {  // from shared memory
    const uint4 v = Shared::ld16(src);
    w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}

// keeps the first n (0 .. 4) bytes of a word / the first n (0 .. 2) half-words
__device__ __forceinline__ uint32_t keep_bytes(uint32_t w, int n) { return n >= 4 ? w : n <= 0 ? 0u : w & ((1u << (8 * n)) - 1u); }
__device__ __forceinline__ uint32_t keep_halves(uint32_t w, int n) { return n >= 2 ? w : n <= 0 ? 0u : w & 0xFFFFu; }

// ---- flags of fine blocks ------------------------------------------------------------------
// bit 7 of every byte of the result tells whether that byte of d is non-zero
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t d) {
    return (((d & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | d) & 0x80808080u;
}
// d0, d1 = new exponents ^ cached exponents of eight consecutive values (one byte each): one flag
// per value, value 0 in bit 0.  The non-zero marks of d0 go to bits 0, 8, 16, 24 and those of d1 to
// bits 4, 12, 20, 28; one multiply then gathers bit 8i into bit 24 + i and bit 8i + 4 into bit
// 28 + i (all partial products land on distinct bits below 32, so nothing carries).
__device__ __forceinline__ uint32_t value_flags8(uint32_t d0, uint32_t d1) {
    const uint32_t t = (nonzero_bytes(d0) >> 7) | (nonzero_bytes(d1) >> 3);
    return (t * 0x01020408u) >> 24;
}
// d = the same for four values: one flag per block of 2^log2b values (log2b = 1, 2: two, one flag)
__device__ __forceinline__ uint32_t word_block_flags(uint32_t d, uint32_t log2b) {
    if (log2b == 1) return ((d & 0xFFFFu) != 0u ? 1u : 0u) | ((d >> 16) != 0u ? 2u : 0u);
    return d != 0u ? 1u : 0u;
}

// The inverse for fine blocks: `flags` = one flag per block of a piece, lowest block first; all bits of the byte
// of every value of a flagged block, for the four values 4 i .. 4 i + 3 of the piece.
__device__ __forceinline__ uint32_t flagged_bytes(uint32_t flags, uint32_t log2b, uint32_t i) {
    if (log2b == 0) return ((((flags >> (4u * i)) & 0xFu) * 0x00204081u) & 0x01010101u) * 0xFFu;
    if (log2b == 1) return (((flags >> (2u * i)) & 1u) * 0xFFFFu) | (((flags >> (2u * i + 1u)) & 1u) * 0xFFFF0000u);
    return ((flags >> (log2b == 2 ? i : i >> 1)) & 1u) * 0xFFFFFFFFu;
}

// ---- pieces --------------------------------------------------------------------------------
template <int DT>
struct Piece;

// bf16: 8 values = 16 B of weights, 8 exponent bytes, 8 sm bytes
template <>
struct Piece<CIERA_BF16> {
    static constexpr int kValues = 8;
    static constexpr int kLog2Values = 3;
    static constexpr int kPerThread = 2;  // pieces per thread
    static constexpr int kExpWords = 2;
    static constexpr int kSmWords = 2;
    static constexpr int kWeightWords = 4;
    // first value (inside the tile) of piece p of consumer thread tid
    static __device__ __forceinline__ uint32_t start(uint32_t tid, int p) {
        return (uint32_t)p * (kTileValues / 2) + tid * 8u;
    }

    uint32_t e[kExpWords];
    uint32_t s[kSmWords];

    template <class M>
    __device__ __forceinline__ void split_full(const uint8_t* w) {
        const uint4 a = M::ld16(w);
        bf16_split4(a.x, a.y, e[0], s[0]);
        bf16_split4(a.z, a.w, e[1], s[1]);
    }
    // the first nvalid (< 8) values; the others read as +0.0 (exponent 0)
    __device__ __forceinline__ void split_partial(const uint8_t* w, int nvalid) {
        uint32_t x[4] = {0, 0, 0, 0};
        const uint16_t* p = reinterpret_cast<const uint16_t*>(w);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < nvalid) x[i >> 1] |= (uint32_t)p[i] << (16 * (i & 1));
        bf16_split4(x[0], x[1], e[0], s[0]);
        bf16_split4(x[2], x[3], e[1], s[1]);
    }
    // the first nvalid values of a whole piece in shared memory; the others read as +0.0 (exponent 0)
    __device__ __forceinline__ void split_first(const uint8_t* w, int nvalid) {
        const uint4 a = Shared::ld16(w);
        bf16_split4(keep_halves(a.x, nvalid), keep_halves(a.y, nvalid - 2), e[0], s[0]);
        bf16_split4(keep_halves(a.z, nvalid - 4), keep_halves(a.w, nvalid - 6), e[1], s[1]);
    }
    template <class M>
    __device__ __forceinline__ void load_exp_full(const uint8_t* src) {
        const uint2 v = M::ld8(src);
        e[0] = v.x; e[1] = v.y;
    }
    template <class M>
    __device__ __forceinline__ void store_exp_full(uint8_t* dst) const { M::st8(dst, make_uint2(e[0], e[1])); }
    __device__ __forceinline__ void load_exp_partial(const uint8_t* src, int nvalid) { load_bytes_partial<8>(e, src, nvalid); }
    // the first nvalid exponents of a whole piece in shared memory; the others read as 0
    __device__ __forceinline__ void load_exp_first(const uint8_t* src, int nvalid) {
        const uint2 v = Shared::ld8(src);
        e[0] = keep_bytes(v.x, nvalid); e[1] = keep_bytes(v.y, nvalid - 4);
    }
    __device__ __forceinline__ void store_exp_partial(uint8_t* dst, int nvalid) const { store_bytes_partial<8>(dst, e, nvalid); }
    template <class M>
    __device__ __forceinline__ void load_sm_full(const uint8_t* src) {
        const uint2 v = M::ld8(src);
        s[0] = v.x; s[1] = v.y;
    }
    template <class M>
    __device__ __forceinline__ void store_sm_full(uint8_t* dst) const { M::st8(dst, make_uint2(s[0], s[1])); }
    __device__ __forceinline__ void load_sm_partial(const uint8_t* src, int nvalid) { load_bytes_partial<8>(s, src, nvalid); }
    __device__ __forceinline__ void store_sm_partial(uint8_t* dst, int nvalid) const { store_bytes_partial<8>(dst, s, nvalid); }
    template <class M>
    __device__ __forceinline__ void merge_store_full(uint8_t* w) const {
        uint4 a;
        bf16_merge4(e[0], s[0], a.x, a.y);
        bf16_merge4(e[1], s[1], a.z, a.w);
        M::st16(w, a);
    }
    __device__ __forceinline__ void merge_store_partial(uint8_t* w, int nvalid) const {
        uint32_t x[4];
        bf16_merge4(e[0], s[0], x[0], x[1]);
        bf16_merge4(e[1], s[1], x[2], x[3]);
        store_halves_partial<8>(w, x, nvalid);
    }
    // the weights at `src` (shared memory) with this piece's exponents in place of their own
    __device__ __forceinline__ void exchange(const uint8_t* src, uint32_t (&w)[kWeightWords]) const {
        load_weights(src, w);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            w[i] = bitselect(0x7F807F80u, __byte_perm(e[i >> 1], 0u, (i & 1) ? 0x4342u : 0x4140u) << 7, w[i]);
    }
    static __device__ __forceinline__ void load_weights(const uint8_t* src, uint32_t (&w)[kWeightWords]) { load_16_bytes(src, w); }
    // the exponents of a piece's weights
    __device__ __forceinline__ void exponents_of(const uint32_t (&w)[kWeightWords]) {
        bf16_split4(w[0], w[1], e[0], s[0]);
        bf16_split4(w[2], w[3], e[1], s[1]);
    }
    template <class M>
    static __device__ __forceinline__ void store_weights(uint8_t* dst, const uint32_t (&w)[kWeightWords]) {
        M::st16(dst, make_uint4(w[0], w[1], w[2], w[3]));
    }
    static __device__ __forceinline__ void store_weights_first(uint8_t* dst, const uint32_t (&w)[kWeightWords], int nvalid) {
        store_halves_partial<8>(dst, w, nvalid);
    }
    __device__ __forceinline__ bool differs(const Piece& o) const { return ((e[0] ^ o.e[0]) | (e[1] ^ o.e[1])) != 0; }
    // one flag per block of 2^log2b values (log2b <= 3), lowest block first
    __device__ __forceinline__ uint32_t block_flags(const Piece& o, uint32_t log2b) const {
        if (log2b >= 3) return differs(o) ? 1u : 0u;
        if (log2b == 0) return value_flags8(e[0] ^ o.e[0], e[1] ^ o.e[1]);
        const uint32_t per_word = 4u >> log2b;
        return word_block_flags(e[0] ^ o.e[0], log2b) | (word_block_flags(e[1] ^ o.e[1], log2b) << per_word);
    }
};

// fp32: 16 values = 64 B of weights, 16 exponent bytes, 48 sm bytes
template <>
struct Piece<CIERA_FP32> {
    static constexpr int kValues = 16;
    static constexpr int kLog2Values = 4;
    static constexpr int kPerThread = 1;
    static constexpr int kExpWords = 4;
    static constexpr int kSmWords = 12;
    static constexpr int kWeightWords = 16;
    static __device__ __forceinline__ uint32_t start(uint32_t tid, int) { return tid * 16u; }

    uint32_t e[kExpWords];
    uint32_t s[kSmWords];

    __device__ __forceinline__ void from_words(const uint32_t* x) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            e[i] = fp32_exp4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]);
            fp32_pack4(fp32_sm(x[4 * i]), fp32_sm(x[4 * i + 1]), fp32_sm(x[4 * i + 2]), fp32_sm(x[4 * i + 3]),
                       s[3 * i], s[3 * i + 1], s[3 * i + 2]);
        }
    }
    template <class M>
    __device__ __forceinline__ void split_full(const uint8_t* w) {
        uint32_t x[16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint4 v = M::ld16(w + 16 * i);
            x[4 * i] = v.x; x[4 * i + 1] = v.y; x[4 * i + 2] = v.z; x[4 * i + 3] = v.w;
        }
        from_words(x);
    }
    __device__ __forceinline__ void split_partial(const uint8_t* w, int nvalid) {
        uint32_t x[16];
        const uint32_t* p = reinterpret_cast<const uint32_t*>(w);
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = i < nvalid ? p[i] : 0u;
        from_words(x);
    }
    // the first nvalid values of a whole piece in shared memory; the others read as +0.0 (exponent 0)
    __device__ __forceinline__ void split_first(const uint8_t* w, int nvalid) {
        uint32_t x[16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint4 v = Shared::ld16(w + 16 * i);
            x[4 * i] = v.x; x[4 * i + 1] = v.y; x[4 * i + 2] = v.z; x[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i >= nvalid) x[i] = 0u;
        from_words(x);
    }
    template <class M>
    __device__ __forceinline__ void load_exp_full(const uint8_t* src) {
        const uint4 v = M::ld16(src);
        e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
    }
    template <class M>
    __device__ __forceinline__ void store_exp_full(uint8_t* dst) const { M::st16(dst, make_uint4(e[0], e[1], e[2], e[3])); }
    __device__ __forceinline__ void load_exp_partial(const uint8_t* src, int nvalid) { load_bytes_partial<16>(e, src, nvalid); }
    // the first nvalid exponents of a whole piece in shared memory; the others read as 0
    __device__ __forceinline__ void load_exp_first(const uint8_t* src, int nvalid) {
        const uint4 v = Shared::ld16(src);
        e[0] = keep_bytes(v.x, nvalid); e[1] = keep_bytes(v.y, nvalid - 4);
        e[2] = keep_bytes(v.z, nvalid - 8); e[3] = keep_bytes(v.w, nvalid - 12);
    }
    __device__ __forceinline__ void store_exp_partial(uint8_t* dst, int nvalid) const { store_bytes_partial<16>(dst, e, nvalid); }
    template <class M>
    __device__ __forceinline__ void load_sm_full(const uint8_t* src) {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const uint4 v = M::ld16(src + 16 * i);
            s[4 * i] = v.x; s[4 * i + 1] = v.y; s[4 * i + 2] = v.z; s[4 * i + 3] = v.w;
        }
    }
    template <class M>
    __device__ __forceinline__ void store_sm_full(uint8_t* dst) const {
#pragma unroll
        for (int i = 0; i < 3; ++i) M::st16(dst + 16 * i, make_uint4(s[4 * i], s[4 * i + 1], s[4 * i + 2], s[4 * i + 3]));
    }
    __device__ __forceinline__ void load_sm_partial(const uint8_t* src, int nvalid) { load_bytes_partial<48>(s, src, 3 * nvalid); }
    __device__ __forceinline__ void store_sm_partial(uint8_t* dst, int nvalid) const { store_bytes_partial<48>(dst, s, 3 * nvalid); }
    __device__ __forceinline__ void merge_words(uint32_t* x) const {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            uint32_t s0, s1, s2, s3;
            fp32_unpack4(s[3 * i], s[3 * i + 1], s[3 * i + 2], s0, s1, s2, s3);
            x[4 * i] = fp32_merge(e[i], s0);
            x[4 * i + 1] = fp32_merge(e[i] >> 8, s1);
            x[4 * i + 2] = fp32_merge(e[i] >> 16, s2);
            x[4 * i + 3] = fp32_merge(e[i] >> 24, s3);
        }
    }
    template <class M>
    __device__ __forceinline__ void merge_store_full(uint8_t* w) const {
        uint32_t x[16];
        merge_words(x);
#pragma unroll
        for (int i = 0; i < 4; ++i) M::st16(w + 16 * i, make_uint4(x[4 * i], x[4 * i + 1], x[4 * i + 2], x[4 * i + 3]));
    }
    __device__ __forceinline__ void merge_store_partial(uint8_t* w, int nvalid) const {
        uint32_t x[16];
        merge_words(x);
        uint32_t* p = reinterpret_cast<uint32_t*>(w);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < nvalid) p[i] = x[i];
    }
    // the weights at `src` (shared memory) with this piece's exponents in place of their own
    __device__ __forceinline__ void exchange(const uint8_t* src, uint32_t (&w)[kWeightWords]) const {
        load_weights(src, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            w[4 * i] = bitselect(0x7F800000u, e[i] << 23, w[4 * i]);
            w[4 * i + 1] = bitselect(0x7F800000u, e[i] << 15, w[4 * i + 1]);
            w[4 * i + 2] = bitselect(0x7F800000u, e[i] << 7, w[4 * i + 2]);
            w[4 * i + 3] = bitselect(0x7F800000u, e[i] >> 1, w[4 * i + 3]);
        }
    }
    static __device__ __forceinline__ void load_weights(const uint8_t* src, uint32_t (&w)[kWeightWords]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) load_16_bytes(src + 16 * i, w + 4 * i);
    }
    // the exponents of a piece's weights
    __device__ __forceinline__ void exponents_of(const uint32_t (&w)[kWeightWords]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = fp32_exp4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
    }
    template <class M>
    static __device__ __forceinline__ void store_weights(uint8_t* dst, const uint32_t (&w)[kWeightWords]) {
#pragma unroll
        for (int i = 0; i < 4; ++i) M::st16(dst + 16 * i, make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]));
    }
    static __device__ __forceinline__ void store_weights_first(uint8_t* dst, const uint32_t (&w)[kWeightWords], int nvalid) {
        uint32_t* const p = reinterpret_cast<uint32_t*>(dst);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (i < nvalid) p[i] = w[i];
    }
    __device__ __forceinline__ bool differs(const Piece& o) const {
        return ((e[0] ^ o.e[0]) | (e[1] ^ o.e[1]) | (e[2] ^ o.e[2]) | (e[3] ^ o.e[3])) != 0;
    }
    // one flag per block of 2^log2b values (log2b <= 3), lowest block first
    __device__ __forceinline__ uint32_t block_flags(const Piece& o, uint32_t log2b) const {
        if (log2b >= 3)
            return (((e[0] ^ o.e[0]) | (e[1] ^ o.e[1])) != 0 ? 1u : 0u) | (((e[2] ^ o.e[2]) | (e[3] ^ o.e[3])) != 0 ? 2u : 0u);
        if (log2b == 0)
            return value_flags8(e[0] ^ o.e[0], e[1] ^ o.e[1]) | (value_flags8(e[2] ^ o.e[2], e[3] ^ o.e[3]) << 8);
        const uint32_t per_word = 4u >> log2b;
        uint32_t f = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) f |= word_block_flags(e[i] ^ o.e[i], log2b) << (per_word * i);
        return f;
    }
};

// fp16: 8 values = 16 B of weights, 8 exponent bytes in the caches, and on the wire 11 bytes of
// sign-plus-mantissa (8 x 11 bits, value j at bits [11 j, 11 j + 11)) and 5 bytes of exponents
// (8 x 5 bits).  Thread -> value layout as for bf16.
template <>
struct Piece<CIERA_FP16> {
    static constexpr int kValues = 8;
    static constexpr int kLog2Values = 3;
    static constexpr int kPerThread = 2;
    static constexpr int kExpWords = 2;
    static constexpr int kWeightWords = 4;
    static __device__ __forceinline__ uint32_t start(uint32_t tid, int p) {
        return (uint32_t)p * (kTileValues / 2) + tid * 8u;
    }

    static constexpr uint32_t kWarpSmBytes = 32u * 11u;  // packed sign-plus-mantissa of a warp's 32 pieces

    uint32_t e[2];  // 8 exponents, one byte each (0..31)
    uint32_t s[3];  // 88 bits of sign-plus-mantissa

    // w = eight fp16 values, two per word
    __device__ __forceinline__ void split_words(const uint32_t w[4]) {
        // p[i] = the two values' 11-bit fields side by side (22 bits): mantissa bits 9:0 stay, the sign
        // (bit 15) moves to bit 10, the second value's mantissa (bits 25:16) to 20:11, its sign (bit 31) to 21
        uint32_t e2[4], p[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t t5 = w[i] >> 5, t10 = w[i] >> 10;
            e2[i] = t10 & 0x001F001Fu;
            p[i] = (w[i] & 0x000003FFu) | (t5 & 0x001FFC00u) | (t10 & 0x00200000u);
        }
        e[0] = __byte_perm(e2[0], e2[1], 0x6420);
        e[1] = __byte_perm(e2[2], e2[3], 0x6420);
        s[0] = p[0] | (p[1] << 22);
        s[1] = (p[1] >> 10) | (p[2] << 12);
        s[2] = (p[2] >> 20) | (p[3] << 2);
    }
    // two values at a time: their exponents to bits 14:10 and 30:26, their fields (bits 21:0) as split_words left them
    __device__ __forceinline__ void merge_words(uint32_t w[4]) const {
        const uint32_t p[4] = {s[0], __funnelshift_r(s[0], s[1], 22), __funnelshift_r(s[1], s[2], 12), s[2] >> 2};
#pragma unroll
        for (int i = 0; i < 4; ++i)
            w[i] = (p[i] & 0x3FFu) | ((p[i] << 5) & 0x03FF8000u) | ((p[i] << 10) & 0x80000000u) | exponent_bits(i);
    }
    // the exponents of values 2 i and 2 i + 1 where they lie in their two values
    __device__ __forceinline__ uint32_t exponent_bits(int i) const {
        return (__byte_perm(e[i >> 1], 0u, (i & 1) ? 0x4342u : 0x4140u) << 10) & 0x7C007C00u;
    }
    // the weights at `src` (shared memory) with this piece's exponents in place of their own
    __device__ __forceinline__ void exchange(const uint8_t* src, uint32_t (&w)[kWeightWords]) const {
        load_weights(src, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i] = (w[i] & 0x83FF83FFu) | exponent_bits(i);
    }
    static __device__ __forceinline__ void load_weights(const uint8_t* src, uint32_t (&w)[kWeightWords]) { load_16_bytes(src, w); }
    // the exponents of a piece's weights
    __device__ __forceinline__ void exponents_of(const uint32_t (&w)[kWeightWords]) { split_words(w); }
    template <class M>
    static __device__ __forceinline__ void store_weights(uint8_t* dst, const uint32_t (&w)[kWeightWords]) {
        M::st16(dst, make_uint4(w[0], w[1], w[2], w[3]));
    }
    static __device__ __forceinline__ void store_weights_first(uint8_t* dst, const uint32_t (&w)[kWeightWords], int nvalid) {
        store_halves_partial<8>(dst, w, nvalid);
    }
    template <class M>
    __device__ __forceinline__ void split_full(const uint8_t* src) {
        const uint4 v = M::ld16(src);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        split_words(w);
    }
    // the first nvalid (< 8) values; the others read as +0.0
    __device__ __forceinline__ void split_partial(const uint8_t* src, int nvalid) {
        const uint16_t* p = reinterpret_cast<const uint16_t*>(src);
        uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < nvalid) w[i >> 1] |= (uint32_t)p[i] << (16 * (i & 1));
        split_words(w);
    }
    // the first nvalid values of a whole piece in shared memory; the others read as +0.0
    __device__ __forceinline__ void split_first(const uint8_t* src, int nvalid) {
        const uint4 v = Shared::ld16(src);
        const uint32_t w[4] = {keep_halves(v.x, nvalid), keep_halves(v.y, nvalid - 2), keep_halves(v.z, nvalid - 4),
                               keep_halves(v.w, nvalid - 6)};
        split_words(w);
    }
    template <class M>
    __device__ __forceinline__ void merge_store_full(uint8_t* dst) const {
        uint32_t w[4];
        merge_words(w);
        M::st16(dst, make_uint4(w[0], w[1], w[2], w[3]));
    }
    __device__ __forceinline__ void merge_store_partial(uint8_t* dst, int nvalid) const {
        uint32_t w[4];
        merge_words(w);
        store_halves_partial<8>(dst, w, nvalid);
    }
    template <class M>
    __device__ __forceinline__ void load_exp_full(const uint8_t* src) {
        const uint2 v = M::ld8(src);
        e[0] = v.x; e[1] = v.y;
    }
    template <class M>
    __device__ __forceinline__ void store_exp_full(uint8_t* dst) const { M::st8(dst, make_uint2(e[0], e[1])); }
    __device__ __forceinline__ void load_exp_partial(const uint8_t* src, int nvalid) { load_bytes_partial<8>(e, src, nvalid); }
    // the first nvalid exponents of a whole piece in shared memory; the others read as 0
    __device__ __forceinline__ void load_exp_first(const uint8_t* src, int nvalid) {
        const uint2 v = Shared::ld8(src);
        e[0] = keep_bytes(v.x, nvalid); e[1] = keep_bytes(v.y, nvalid - 4);
    }
    __device__ __forceinline__ void store_exp_partial(uint8_t* dst, int nvalid) const { store_bytes_partial<8>(dst, e, nvalid); }
    __device__ __forceinline__ bool differs(const Piece& o) const { return ((e[0] ^ o.e[0]) | (e[1] ^ o.e[1])) != 0; }
    // one flag per block of 2^log2b values (log2b <= 3), lowest block first (the exponents lie one byte each, as for bf16)
    __device__ __forceinline__ uint32_t block_flags(const Piece& o, uint32_t log2b) const {
        if (log2b >= 3) return differs(o) ? 1u : 0u;
        if (log2b == 0) return value_flags8(e[0] ^ o.e[0], e[1] ^ o.e[1]);
        const uint32_t per_word = 4u >> log2b;
        return word_block_flags(e[0] ^ o.e[0], log2b) | (word_block_flags(e[1] ^ o.e[1], log2b) << per_word);
    }

    // the 8 exponents as 40 bits: low word and high byte (four bytes of 5 bits -> two fields of 10 -> one of 20)
    __device__ __forceinline__ void pack_exponents(uint32_t& lo, uint32_t& hi) const {
        uint32_t z[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t v = (e[i] & 0x001F001Fu) | ((e[i] >> 3) & 0x03E003E0u);
            z[i] = (v & 0x3FFu) | ((v >> 6) & 0xFFC00u);
        }
        lo = z[0] | (z[1] << 20);
        hi = z[1] >> 12;
    }
    __device__ __forceinline__ void unpack_exponents(uint32_t lo, uint32_t hi) {
        const uint32_t z[2] = {lo, (lo >> 20) | (hi << 12)};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const uint32_t v = (z[i] & 0x3FFu) | ((z[i] << 6) & 0x03FF0000u);
            e[i] = (v & 0x001F001Fu) | ((v << 3) & 0x1F001F00u);
        }
    }
    // the packed exponents of a whole piece from shared memory (any alignment): the two words that hold the 5 bytes
    __device__ __forceinline__ void load_packed_exponents(const uint8_t* src) {
        const uint32_t skew = (uint32_t)reinterpret_cast<uintptr_t>(src) & 3u;
        const uint32_t w0 = Shared::ld4(src - skew), w1 = Shared::ld4(src - skew + 4);
        unpack_exponents(__funnelshift_r(w0, w1, 8u * skew), w1 >> (8u * skew));
    }
    // the packed exponents of the piece from `src` (5 bytes, any alignment; nvalid < 8: fewer)
    template <class M>
    __device__ __forceinline__ void load_packed_exponents(const uint8_t* src, int nvalid) {
        const int nbytes = (5 * nvalid + 7) >> 3;
        uint32_t lo = 0, hi = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            if (i < nbytes) {
                const uint32_t b = M::ld1(src + i);
                if (i < 4)
                    lo |= b << (8 * i);
                else
                    hi = b;
            }
        }
        unpack_exponents(lo, hi);
    }

    // Packed sign-plus-mantissa of a piece in a section whose pieces are all complete: the four lanes
    // 4k..4k+3 share 44 bytes = 11 aligned words, lane a holds bits [88a, 88a+88) of them.
    // `section` = start of the tile's part of the section, `piece` = index of the piece in the tile.
    template <class M>
    __device__ __forceinline__ void load_sm_group(const uint8_t* section, uint32_t piece, uint32_t lane) {
        const uint32_t a = lane & 3u;
        // lane a's bits start at word {0, 2, 5, 8}, bit {0, 24, 16, 8} of the group
        const uint32_t first = (11u * a) >> 2, sh = (88u * a) & 31u;
        const uint8_t* src = section + (size_t)11 * (piece - a) + 4u * first;
        const uint32_t w0 = M::ld4(src), w1 = M::ld4(src + 4), w2 = M::ld4(src + 8);
        const uint32_t w3 = (a == 0u || a == 3u) ? 0u : M::ld4(src + 12);  // lanes 0 and 3 end inside their third word
        s[0] = sh ? (w0 >> sh) | (w1 << (32u - sh)) : w0;
        s[1] = sh ? (w1 >> sh) | (w2 << (32u - sh)) : w1;
        s[2] = (sh ? (w2 >> sh) | (w3 << (32u - sh)) : w2) & 0x00FFFFFFu;
    }
    // lane a writes words 3a, 3a+1, 3a+2 of the group (lane 3: two words), taking the low bits of the
    // next lane's first word where its own bits end inside a word.  All 32 lanes call this.
    __device__ __forceinline__ void store_sm_group(uint8_t* section, uint32_t piece, uint32_t lane) const {
        const uint32_t a = lane & 3u, sh = 8u * a;
        const uint32_t next0 = __shfl_down_sync(0xffffffffu, s[0], 1);
        uint32_t* dst = reinterpret_cast<uint32_t*>(section + (size_t)11 * (piece - a)) + 3u * a;
        dst[0] = __funnelshift_r(s[0], s[1], sh);
        dst[1] = __funnelshift_r(s[1], s[2], sh);
        if (a != 3u) dst[2] = (s[2] >> sh) | (next0 << (24u - sh));
    }
    // The same for the warp's 32 pieces by way of 352 bytes of shared memory (`gather`, 16-byte aligned), from which
    // 22 lanes write 16 bytes each, and again `twin` bytes further on.
    __device__ __forceinline__ void store_sm_warp(uint8_t* section, uint32_t piece, uint8_t* gather, int64_t twin, uint32_t lane) const {
        store_sm_group(gather, lane, lane);
        __syncwarp();
        if (lane < kWarpSmBytes / 16u) {
            const uint4 v = ld_shared16(gather + 16u * lane);
            uint8_t* const dst = section + (size_t)11 * (piece - lane) + 16u * lane;
            st_stream16(dst, v);
            st_stream16(dst + twin, v);
        }
        __syncwarp();  // the gather space is free again
    }
    // byte by byte (pieces of a tile with a ragged end)
    __device__ __forceinline__ void load_sm_bytes(const uint8_t* src, int nvalid) {
        s[0] = s[1] = s[2] = 0;
        const int nbytes = (11 * nvalid + 7) >> 3;
        for (int i = 0; i < nbytes; ++i) s[i >> 2] |= (uint32_t)src[i] << (8 * (i & 3));
    }
    __device__ __forceinline__ void store_sm_bytes(uint8_t* dst, int nvalid) const {
        const int nbytes = (11 * nvalid + 7) >> 3;
        for (int i = 0; i < nbytes; ++i) dst[i] = (uint8_t)(s[i >> 2] >> (8 * (i & 3)));
    }
};

// number of valid values of the piece starting at value `start` in a tile of nv values
template <int DT>
__device__ __forceinline__ int piece_valid(uint32_t start, uint32_t nv) {
    return start >= nv ? 0 : (int)min((uint32_t)Piece<DT>::kValues, nv - start);
}

// Block flags of a tile from the vote bits "my piece differs" (one warp).  `pl2` = log2 of the
// values per piece.  Fills bm (one bit per block of the tile) and pre (set bits before each word);
// returns the number of changed blocks of the tile.
__device__ __forceinline__ uint32_t build_block_bitmap(const uint32_t* ballot, uint32_t* bm, uint16_t* pre,
                                                       uint32_t log2b, uint32_t pl2, uint32_t lane) {
    const uint32_t gl2 = log2b - pl2;           // log2(pieces per block)
    const uint32_t nbt = kTileValues >> log2b;  // blocks of a full tile
    if (nbt > 32 && gl2 >= 1) {
        // More than one word of block flags (2 to 16 pieces per block): lane l turns vote word l into
        // its 32 >> gl2 block flags -- fold the votes of a block onto its first bit, gather those bits --
        // the 2^gl2 lanes whose flags share a word of bm combine them, and one scan does for the tile.
        const uint32_t vote_words = (uint32_t)kTileValues >> (pl2 + 5);  // 32 or 16
        uint32_t t = lane < vote_words ? ballot[lane] : 0u;
        for (uint32_t k = 0; k < gl2; ++k) t |= t >> (1u << k);
        const uint32_t cnt = 32u >> gl2;
        uint32_t fl = 0;
        for (uint32_t j = 0; j < cnt; ++j) fl |= ((t >> (j << gl2)) & 1u) << j;
        uint32_t v = fl << ((lane * cnt) & 31u);
        for (uint32_t k = 0; k < gl2; ++k) v |= __shfl_xor_sync(0xffffffffu, v, 1u << k);
        const uint32_t nwords = nbt >> 5;  // 2 .. 16
        uint32_t word = __shfl_sync(0xffffffffu, v, (lane << gl2) & 31u);
        if (lane >= nwords) word = 0u;
        const uint32_t pc = __popc(word);
        uint32_t incl = pc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if ((int)lane >= o) incl += u;
        }
        if (lane < nwords) {
            bm[lane] = word;
            pre[lane] = (uint16_t)(incl - pc);
        }
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        __syncwarp();
        return total;
    }
    uint32_t run = 0;
    for (uint32_t base = 0; base < nbt; base += 32) {
        const uint32_t i = base + lane;
        bool f = false;
        if (i < nbt) {
            const uint32_t g0 = i << gl2;
            if (gl2 <= 5) {
                const uint32_t width = 1u << gl2;
                const uint32_t m = width == 32 ? 0xffffffffu : ((1u << width) - 1u);
                f = ((ballot[g0 >> 5] >> (g0 & 31)) & m) != 0;
            } else {
                const uint32_t nw = 1u << (gl2 - 5);
                uint32_t acc = 0;
                for (uint32_t j = 0; j < nw; ++j) acc |= ballot[(g0 >> 5) + j];
                f = acc != 0;
            }
        }
        const uint32_t word = __ballot_sync(0xffffffffu, f);
        if (lane == 0) {
            bm[base >> 5] = word;
            pre[base >> 5] = (uint16_t)run;
        }
        run += __popc(word);
    }
    __syncwarp();
    return run;
}

__device__ __forceinline__ TileDesc load_tile_desc(const TileDesc* t) {
    const uint4* p = reinterpret_cast<const uint4*>(t);
    uint4 a = __ldg(p), b = __ldg(p + 1), c = __ldg(p + 2);
    TileDesc d;
    d.w_off = (uint64_t)a.x | ((uint64_t)a.y << 32);
    d.c_off = (uint64_t)a.z | ((uint64_t)a.w << 32);
    d.msg_off = (uint64_t)b.x | ((uint64_t)b.y << 32);
    d.n_unit = (uint64_t)b.z | ((uint64_t)b.w << 32);
    d.unit = c.x;
    d.tile_in_unit = c.y;
    d.first_tile = c.z;
    d.n_tiles_unit = c.w;
    return d;
}

}  // namespace ciera
