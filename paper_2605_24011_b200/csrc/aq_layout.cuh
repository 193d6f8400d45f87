// Device-private weight layout ("fragment layout") and the bit tricks that read it.
//
// The canonical container (Appendix D) is row-major block records; on the
// device the same bits are regrouped so that one warp reads what one tensor
// core instruction needs with 16-byte accesses, and so that a code can be used
// as a tensor-core operand WHERE IT LIES, with one AND and no shift:
//
//   fragment = 16 rows x 128 k (4 blocks of 32), FB = 256 (bits+1) bytes
//     bytes [0,256)  : half2 (scale, min) at [row r][block j] -> (r*4 + j)*4
//     bytes [256,FB) : codes.  Slot s = g*4 + t (g = row mod 8, t = 0..3) owns,
//                      for rows g and g+8 and each block j, the 8 codes
//                      8t .. 8t+7 of that block.
//   order    = [k-slab S][row tile R] ; N padded to 16, K to 256.  The fragments of
//              neighbouring row tiles are contiguous: 128 rows x 128 k, what a tensor
//              core instruction of 128 rows wants, is one copy of 8 fragments.
//   unit     = the fragments of k-slabs 2P and 2P+1 of one row tile.
//
// A slot's 64 codes are 16 groups of 4: group (j, hi, h) = codes 4h .. 4h+3 of the
// slot's block j, row half hi.  The four codes of a group sit in the four bytes of
// ONE word at the SAME bit position pos(j, h), in the byte order 0, 2, 1, 3: a mask
// gives four 8-bit operands, and the low (or, after a shift by 8, the high) bytes of
// the two half words give a pair of k-adjacent codes as two 16-bit operands.  Either
// way the operand is 2^pos * q, and the power of two is taken out elsewhere.
//   4-bit: word 2j + hi, pos 4h.
//   2-bit: word 2 (j & 1) + hi, pos 4h + 2 (j >> 1).
//   3-bit: word 2j + hi, pos 4h for j < 3; the words of j = 3 are spread over the
//          free bits 3 and 7 of every byte: bit b of word 6 + x, pos 4h, is bit
//          3 + 4h of word 3x + b.
//   words 0..3 lie at 256 + s*16; words 4.. at 768 + s*8 (3-bit) or 768 + s*16.
#pragma once
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace aq {

constexpr int ROWS = 16;        // rows per fragment
constexpr int SLAB = 128;       // k per fragment
constexpr int SCALE_BYTES = 256;

__host__ __device__ constexpr int frag_bytes(int bits) { return 256 * (bits + 1); }
__host__ __device__ constexpr int64_t frag_index(int64_t S, int64_t R, int64_t NT) { return S * NT + R; }

// Home of bit tb of code c (0..7) of the slot's block j, row half hi: the index
// of the slot's 32-bit word and the bit position in it.
__host__ __device__ inline void slot_bit_home(int bits, int j, int hi, int c, int tb, int& widx, int& bitpos) {
    const int h = c >> 2;
    const int byte = (c & 1) * 2 + ((c >> 1) & 1);   // codes 0, 1, 2, 3 of a group: bytes 0, 2, 1, 3
    if (bits == 2) {
        widx = 2 * (j & 1) + hi; bitpos = 8 * byte + 4 * h + 2 * (j >> 1) + tb;
    } else if (bits == 4 || j < 3) {
        widx = 2 * j + hi; bitpos = 8 * byte + 4 * h + tb;
    } else {
        widx = 3 * hi + tb; bitpos = 8 * byte + 4 * h + 3;
    }
}

// Byte offset, inside the fragment, of word widx of slot s.
__host__ __device__ inline int slot_word_offset(int bits, int s, int widx) {
    if (bits == 2) return 256 + s * 16 + widx * 4;
    if (bits == 4) return 256 + (widx >> 2) * 512 + s * 16 + (widx & 3) * 4;
    return widx < 4 ? 256 + s * 16 + widx * 4 : 256 + 512 + s * 8 + (widx - 4) * 4;
}

// ---- register-level extraction -------------------------------------------
// A lane's code words for one fragment.
template <int BITS> struct LaneCodes { uint32_t w[2 * BITS]; };

template <int BITS>
__device__ __forceinline__ void load_lane_codes(LaneCodes<BITS>& lc, const uint8_t* frag, int lane) {
    const uint4 a = *reinterpret_cast<const uint4*>(frag + 256 + lane * 16);
    lc.w[0] = a.x; lc.w[1] = a.y; lc.w[2] = a.z; lc.w[3] = a.w;
    if constexpr (BITS == 3) {
        const uint2 b = *reinterpret_cast<const uint2*>(frag + 256 + 512 + lane * 8);
        lc.w[4] = b.x; lc.w[5] = b.y;
    }
    if constexpr (BITS == 4) {
        const uint4 b = *reinterpret_cast<const uint4*>(frag + 256 + 512 + lane * 16);
        lc.w[4] = b.x; lc.w[5] = b.y; lc.w[6] = b.z; lc.w[7] = b.w;
    }
}

__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t mask, uint32_t orv) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(mask), "r"(orv));   // (a & mask) | orv
    return d;
}

// The words the groups are read from: the lane's own ones, for 3 bits with the two spread words gathered behind them.
template <int BITS> struct SlotWords {
    static constexpr int N = BITS == 2 ? 4 : 8;
    uint32_t w[N];
    __device__ __forceinline__ void gather(const LaneCodes<BITS>& lc) {
#pragma unroll
        for (int i = 0; i < 2 * BITS; ++i) w[i] = lc.w[i];
        if constexpr (BITS == 3) {
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                const uint32_t* T = lc.w + 3 * x;
                uint32_t v = (T[0] >> 3) & 0x11111111u;
                v = lop3_and_or(T[1] >> 2, 0x22222222u, v);
                w[6 + x] = lop3_and_or(T[2] >> 1, 0x44444444u, v);
            }
        }
    }
    static __device__ __forceinline__ constexpr int word(int j, int hi) { return BITS == 2 ? 2 * (j & 1) + hi : 2 * j + hi; }
    static __device__ __forceinline__ constexpr int pos(int j, int h) { return BITS == 2 ? 4 * h + 2 * (j >> 1) : 4 * h; }
};

// Pair i (codes 2i, 2i+1) of block j, row half hi (0: row g, 1: row g+8): the
// two codes land in bits [0,BITS) and [16,16+BITS) of the result, OR-ed with
// `orv` (0 for plain integers, a floating-point exponent pattern otherwise).
template <int BITS>
__device__ __forceinline__ uint32_t code_pair(const SlotWords<BITS>& sw, int j, int hi, int i, uint32_t orv) {
    constexpr uint32_t MASK = (1u << BITS) - 1u;
    return lop3_and_or(sw.w[sw.word(j, hi)] >> (8 * (i & 1) + sw.pos(j, i >> 1)), MASK | (MASK << 16), orv);
}

// ---- in-place reader (fp16 operands) ----------------------------------------
// A code left at bit position s of a half-word, everything else masked away,
// IS the binary16 subnormal q * 2^(s - 24) as long as s + BITS <= 10.  One AND
// per A register; a byte shift of the whole word brings the other pair of its
// group into place.  A register r = hi + 2 (i & 1) of instruction f = 2j + h is
// pair i = 2h + (r >> 1) of block j, row half hi.
template <int BITS> struct InPlace {
    static constexpr int NCLS = BITS == 2 ? 4 : 2;           // bit positions 0,2,4,6 / 0,4
    uint32_t w[SlotWords<BITS>::N], w8[SlotWords<BITS>::N];
    __device__ __forceinline__ void prepare(const LaneCodes<BITS>& lc) {
        SlotWords<BITS> sw;
        sw.gather(lc);
#pragma unroll
        for (int i = 0; i < SlotWords<BITS>::N; ++i) { w[i] = sw.w[i]; w8[i] = sw.w[i] >> 8; }
    }
    static __device__ __forceinline__ constexpr int pos(int f) { return SlotWords<BITS>::pos(f >> 1, f & 1); }
    static __device__ __forceinline__ constexpr int cls(int f) { return BITS == 2 ? pos(f) / 2 : pos(f) / 4; }
    static __device__ __forceinline__ constexpr int cls_pos(int c) { return BITS == 2 ? 2 * c : 4 * c; }
    __device__ __forceinline__ uint32_t reg(int f, int r) const {
        constexpr uint32_t MASK = ((1u << BITS) - 1u) * 0x00010001u;
        const int k = SlotWords<BITS>::word(f >> 1, r & 1);
        return ((r >> 1) ? w8[k] : w[k]) & (MASK << pos(f));
    }
    __device__ __forceinline__ uint32_t reg_or(int f, int r, uint32_t orv) const {
        constexpr uint32_t MASK = ((1u << BITS) - 1u) * 0x00010001u;
        const int k = SlotWords<BITS>::word(f >> 1, r & 1);
        return lop3_and_or((r >> 1) ? w8[k] : w[k], MASK << pos(f), orv);
    }
};

}  // namespace aq
