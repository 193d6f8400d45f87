// Device code of the decode kernel's arithmetic (fifth-generation tensor cores; codes and sums in TMEM).
//
// With w = d q + m per block (Eq. 1),   sum_k x w = d * sum q x  +  m * sum x.   The work is cut into halves of units: 128
// rows x 128 k = the eight fragments (16 rows x 128 k) of eight neighbouring row tiles.
//
//   A  = the codes in TMEM, one lane per row.  Lane (g, t) of a warp holds, for rows g and g + 8, the 64 codes of its slot
//        (aq_layout.cuh), which is how tcgen05.st.16x128b takes registers: one AND per register, no shared memory in
//        between.
//   B  = the tokens in shared memory, K-major without swizzle.
//   D  = sums in TMEM, read back one row per lane; the block scales need a sum per block.
//
// One token (kind::i8, exact integers).  Every byte of an A register is a code times 2^pos (pos 0 or 2 for the first group
// of a block's slot, 4 or 6 for the second).  x enters as a block-wise fixed-point number in four signed bytes: scaled by the
// power of two that brings the largest magnitude of its block of 32 into [2^29, 2^30), the elements that meet second groups
// by 2^-4 of that.  So an element is off by at most 2^-30 of that magnitude in a first group and 2^-26 in a second, and
// a binary16 value is exact unless it is 2^19 / 2^15 times smaller (bfloat16: 2^22 / 2^18).  (Blocks below 2^-93, which only
// bfloat16 has: steps of 2^-123 / 2^-119.)  That is below what binary32 sums of the block's products lose, unless the largest
// element meets a weight that decodes to 0.  B = four byte planes of a block in four rows: a chunk of 16 k is 128 bytes, 4 rows of data and 4 of zeros.  The
// instruction of an odd block reads its chunks through a window moved down by 64 bytes, so the planes land in rows 4..7:
// two blocks share one accumulator of 8 columns [block parity][plane].
//
// Several tokens (kind::f16).  A code at bit position s of a half word IS the binary16 subnormal q 2^(s - 24); tensor
// cores take subnormals exactly (but see dt_unpack).  bfloat16 subnormals would push the products below the binary32 normal range: there
// codes are shifted down and OR-ed into the mantissa of 128.0, and  sum x w = d * sum (128 + q) x + (m - 128 d) * sum x.
// B: a chunk of 8 k is 128 bytes, row = token.  Instruction f = 2 j + h (block j, half h of it) reads chunks 2 f and
// 2 f + 1; element 2 t + e of chunk 2 f + c is x[32 j + 8 t + 4 h + 2 c + e].  One accumulator of 16 columns per block:
// columns 0..7 are the tokens' sums of half 0 (the second group of eight B rows is then a region of zeros), 8..15
// those of half 1 (the first group is); they are joined when they are read.  (Joined by the tensor core, which leaves half the
// columns to be read, sums come out up to 1.08 times further from 64 bits for normal activations, 1.5 for heavy-tailed ones.)
//
// Why tcgen05 with so few tokens: with A in TMEM a 128 x 8 x 32 byte or 128 x 16 x 16 half-word instruction takes 8.4 / 9.6
// cycles of the tensor pipe (measured), 8.4 / 19 per 4096 weights, against 117 for the same weights as mma.sync, and one
// thread issues it for four warps.  What is left per 4096 weights at one token is 32 (3 bits: 56) integer instructions, two
// TMEM stores (16x128b: 490 B per clock and SM, the 16x256b form 250) and about 40 instructions that read the sums back.
#pragma once
#include "aq_layout.cuh"
#include "aq_tc.cuh"
#include "aq_tmem.cuh"

namespace aq {

constexpr int DT_ROWS = 128;            // rows of a unit
constexpr int DT_CHUNK = 128;           // bytes of a staged chunk
constexpr int DT_ZERO_BYTES = 256;      // a pair of core matrices of zeros

template <int MT> struct DtShape {      // several tokens
    static constexpr int A_COLS = 64, D_COLS = 64;                 // TMEM columns of half a unit
    static constexpr int X_BYTES = 32 * DT_CHUNK;                  // staged bytes of a slab; then [8 blocks][8 tokens] sums of x
};
template <> struct DtShape<1> {
    static constexpr int A_COLS = 32, D_COLS = 16;
    static constexpr int X_BYTES = 16 * DT_CHUNK;                  // then [8 blocks](sum of x, step of the fixed-point x)
};
template <int MT> constexpr int DT_SUMS = DtShape<MT>::X_BYTES;                           // byte offset of the sums in a staged slab
constexpr int dt_slab_bytes(int M) { return M == 1 ? 2048 + 128 : 4096 + 256; }          // (multiples of 128)

constexpr uint32_t DT_IDESC_I8 = (2u << 4) | (1u << 10) | ((8u >> 3) << 17) | ((uint32_t)(DT_ROWS >> 4) << 24);    // u8 x s8 -> s32, 128 x 8
constexpr uint32_t DT_IDESC_F16 = (1u << 4) | ((16u >> 3) << 17) | ((uint32_t)(DT_ROWS >> 4) << 24);   // f16 x f16 -> f32, 128 x 16
constexpr uint32_t DT_IDESC_BF16 = DT_IDESC_F16 | (1u << 7) | (1u << 10);

// A in TMEM, B in shared memory
__device__ __forceinline__ void umma_i8_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, float* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, int (&v)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
                   "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16f(uint32_t taddr, float* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]), "=f"(v[9]),
                   "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]) : "r"(taddr) : "memory");
}
// two binary32 numbers in a register pair, and a multiply-add on both
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pair2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpair2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// K-major without swizzle: core matrices of 8 rows x 16 bytes, `lbo` apart along K, `sbo` apart along the rows.
__device__ __forceinline__ uint64_t dt_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) | ((uint64_t)1 << 46);
}

// ---- staging of four consecutive elements k .. k + 3 (k a multiple of 4, 0 .. 252) of a slab ----------------------------
// several tokens: two pairs of half words (r: the rounded values)
__device__ __forceinline__ void dt_stage4(uint8_t* slab, int tok, int k, uint2 r) {
    uint8_t* p = slab + ((k >> 5) * 4 + ((k >> 2) & 1) * 2) * DT_CHUNK + tok * 16 + ((k >> 3) & 3) * 4;
    *reinterpret_cast<uint32_t*>(p) = r.x;
    *reinterpret_cast<uint32_t*>(p + DT_CHUNK) = r.y;
}
// one token: the bit pattern of the power of two that brings magnitudes up to `mx` (the block's largest) below 2^30
__device__ __forceinline__ uint32_t dt_fix_scale(float mx) {
    const uint32_t e = __float_as_uint(mx) >> 23;      // biased exponent, mx < 2^(e - 126)
    return min(283u - e, 250u) << 23;
}
// ... and its reciprocal.  A block with an infinity: the conversion to an integer saturates, the digits of 2^31 - 1 and of -2^31
// both stand for about -2^31, and finite elements (below 2^98) come out as 0.  The step is then minus the (infinite) sum: step times a
// sum of codes has the sign it should have, or is NaN where the code is 0, as the product with an infinity is.
__device__ __forceinline__ float dt_fix_step(uint32_t scale_bits, float sum) {
    uint32_t step = (254u << 23) - scale_bits;
    // (written out: a 7B pass takes 835 us with this select, 838 to 840 as a conditional expression, 830 without either)
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %1, %2;\n\tselp.b32 %0, %3, %0, p;\n\t}"
                 : "+r"(step) : "r"(scale_bits), "n"((283u - 255u) << 23), "r"(__float_as_uint(sum) ^ 0x80000000u));
    return __uint_as_float(step);
}
__device__ __forceinline__ void dt_stage4_fix(uint8_t* slab, int k, const float4& v, uint32_t scale_bits) {
    const int h = (k >> 2) & 1;
    const float sc = __uint_as_float(scale_bits - (uint32_t)(h * (4 << 23)));
    // signed bytes: adding 128 to each lower byte, carries included, and taking it out again without them
    auto digits = [&](float x) { return ((uint32_t)__float2int_rn(x * sc) + 0x00808080u) ^ 0x00808080u; };
    const uint32_t a = digits(v.x), b = digits(v.y), c = digits(v.z), d = digits(v.w);
    // 4 x 4 byte transpose; the bytes of a plane in the order 0, 2, 1, 3 of the elements
    const uint32_t ac01 = __byte_perm(a, c, 0x5140), bd01 = __byte_perm(b, d, 0x5140);   // a0 c0 a1 c1, b0 d0 b1 d1
    const uint32_t ac23 = __byte_perm(a, c, 0x7362), bd23 = __byte_perm(b, d, 0x7362);
    uint8_t* p = slab + ((k >> 5) * 2 + h) * DT_CHUNK + ((k >> 3) & 3) * 4;
    *reinterpret_cast<uint32_t*>(p) = __byte_perm(ac01, bd01, 0x5410);
    *reinterpret_cast<uint32_t*>(p + 16) = __byte_perm(ac01, bd01, 0x7632);
    *reinterpret_cast<uint32_t*>(p + 32) = __byte_perm(ac23, bd23, 0x5410);
    *reinterpret_cast<uint32_t*>(p + 48) = __byte_perm(ac23, bd23, 0x7632);
}

// Several tokens, binary16: codes of a first group (half 0) are moved up to the bit position of the second.  The tensor core
// aligns products by the exponents of its operands, the leading zeros of a subnormal included, and drops what lies below: left
// where they lie, codes at position 0 lose up to 8 bits.  Root mean square of the error over sum |x w|, 8 tokens, 4096 columns,
// at 2 / 3 / 4 bits: 4.6e-8 / 3.3e-8 / 1.9e-8 where they lie, 2.8e-9 / 2.7e-9 / 2.8e-9 here (mma.sync, where they lie: 3.0e-8 / 2.6e-8 / 1.9e-8).

// ---- codes -> A registers -------------------------------------------------------------------------------------------
// A lane's slot of one fragment as A registers in tcgen05.st.16x128b order.
template <int BITS, bool BF16>
__device__ __forceinline__ void dt_unpack(const LaneCodes<BITS>& lc, uint32_t (&v)[32]) {
    constexpr uint32_t MAGIC = 0x43004300u;   // bf16 128.0 in both halves
    if constexpr (BF16) {
        SlotWords<BITS> sw;
        sw.gather(lc);
#pragma unroll
        for (int f = 0; f < 8; ++f)
#pragma unroll
            for (int r = 0; r < 4; ++r) v[4 * f + r] = code_pair<BITS>(sw, f >> 1, r & 1, 2 * (f & 1) + (r >> 1), MAGIC);
    } else {
        SlotWords<BITS> sw;
        sw.gather(lc);
#pragma unroll
        for (int f = 0; f < 8; ++f)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t w = sw.w[sw.word(f >> 1, r & 1)], MASK = ((1u << BITS) - 1u) * 0x00010001u;
                const uint32_t x = (f & 1) ? (r < 2 ? w : w >> 8) : (r < 2 ? w << 4 : w >> 4);
                v[4 * f + r] = x & (MASK << sw.pos(f >> 1, 1));
            }
    }
}
template <int BITS, bool BF16>
__device__ __forceinline__ void dt_unpack(const LaneCodes<BITS>& lc, uint32_t (&v)[16]) {
    SlotWords<BITS> sw;
    sw.gather(lc);
    constexpr uint32_t MASK = ((1u << BITS) - 1u) * 0x01010101u;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int hi = 0; hi < 2; ++hi) v[4 * j + 2 * h + hi] = sw.w[sw.word(j, hi)] & (MASK << sw.pos(j, h));
}
// Two fragments at once.
template <int BITS>
__device__ __forceinline__ void dt_unpack2(const uint8_t* frags, int lane, uint32_t (&va)[16], uint32_t (&vb)[16]) {
    LaneCodes<BITS> la, lb;
    load_lane_codes<BITS>(la, frags, lane);
    load_lane_codes<BITS>(lb, frags + frag_bytes(BITS), lane);
    dt_unpack<BITS, false>(la, va);
    dt_unpack<BITS, false>(lb, vb);
}

// ---- a unit's instructions (one elected thread) -----------------------------------------------------------------------
// x: the staged slab; zlow, zhigh: regions of zeros below and above every staged slab.  Descriptors differ by constants:
// the start address is the low field (in 16 bytes), the stride between row groups starts at bit 32.
template <int MT, bool BF16>
__device__ __forceinline__ void dt_issue(uint32_t tmem_a, uint32_t tmem_d, uint32_t x, uint32_t zlow, uint32_t zhigh) {
    constexpr int STEP = 2 * DT_CHUNK / 16;
    if constexpr (MT == 1) {
        const uint64_t bd = dt_desc(x, DT_CHUNK, DT_CHUNK);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            umma_i8_ts(tmem_d + 8 * (j >> 1), tmem_a + 8 * j, bd + (uint64_t)(STEP * j - 4 * (j & 1)), DT_IDESC_I8, (uint32_t)(j & 1));
    } else {
        const uint64_t lo = dt_desc(x, DT_CHUNK, zhigh - x), hi = dt_desc(zlow, DT_CHUNK, x - zlow);
#pragma unroll
        for (int f = 0; f < 16; ++f) {
            const uint64_t bd = (f & 1) ? hi + ((uint64_t)(STEP * f) << 32) : lo + (uint64_t)(STEP * f) - ((uint64_t)(STEP * f) << 32);
            umma_f16_ts(tmem_d + 16 * (f >> 1), tmem_a + 8 * f, bd, BF16 ? DT_IDESC_BF16 : DT_IDESC_F16, (uint32_t)(f & 1));
        }
    }
}

// ---- sums -> the lane's row -----------------------------------------------------------------------------------------
// acc[token] += sum over the unit's 8 blocks of d * (sum q x) + m * (sum x).  dm0, dm1: the row's (scale, min) pairs of
// the two halves; sums: see DtShape.
template <int BITS, int MT, bool BF16>
__device__ __forceinline__ void dt_collect(uint32_t tmem_d, const uint4& dm0, const uint4& dm1, const float* sums, float (&acc)[MT]) {
    const uint32_t w[8] = {dm0.x, dm0.y, dm0.z, dm0.w, dm1.x, dm1.y, dm1.z, dm1.w};
    if constexpr (MT == 1) {
        int v[2][16];
        tmem_ld16(tmem_d, v[0]);
        tmem_ld16(tmem_d + DtShape<1>::D_COLS, v[1]);
        float part[2] = {0.f, 0.f};   // (two chains of multiply-adds)
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) { asm volatile("" : "+r"(v[0][i])); asm volatile("" : "+r"(v[1][i])); }   // (read only after the wait)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            // four planes of a block: |plane| < 2^20, so two of them join exactly in 32 bits
            const int* q = v[j >> 2] + 4 * (j & 3);
            const float lo = (float)(q[1] * 256 + q[0]), hi = (float)(q[3] * 256 + q[2]);
            const float2 xs = *reinterpret_cast<const float2*>(sums + 2 * j);   // sum of x, step of the fixed-point x
            constexpr float unpos[2] = {1.f, 1.f / (float)(1 << SlotWords<BITS>::pos(2, 0))};
            const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
            part[j & 1] = fmaf(p.x * (xs.y * unpos[(j & 3) >> 1]), fmaf(hi, 65536.f, lo), fmaf(p.y, xs.x, part[j & 1]));
        }
        acc[0] += part[0] + part[1];
    } else {
        auto unpos = [](int j) -> float { return BF16 ? 1.f : (float)(1u << (24 - SlotWords<BITS>::pos(j, 1))); };   // a code's power of two
        // BB blocks at a time, [block][half][token]; the next ones' sums are on their way meanwhile
        constexpr int BB = MT == 8 ? 1 : 2;
        float v[2][BB * 2 * MT];
        auto load = [&](int j, float* b) {
#pragma unroll
            for (int i = 0; i < BB; ++i) {
                const uint32_t t = tmem_d + 16 * (j + i);
                if constexpr (MT == 2) { tmem_ld2(t, b + 4 * i); tmem_ld2(t + 8, b + 4 * i + 2); }
                else if constexpr (MT == 4) { tmem_ld4(t, b + 8 * i); tmem_ld4(t + 8, b + 8 * i + 4); }
                else tmem_ld16f(t, b);
            }
        };
        f32x2 a[MT / 2];   // token pairs: one multiply-add instruction for two
#pragma unroll
        for (int m = 0; m < MT / 2; ++m) a[m] = pair2(acc[2 * m], acc[2 * m + 1]);
        load(0, v[0]);
#pragma unroll
        for (int j = 0; j < 8; j += BB) {
            float (&b)[BB * 2 * MT] = v[(j / BB) & 1];
            tmem_ld_wait();
#pragma unroll
            for (int m = 0; m < BB * 2 * MT; ++m) asm volatile("" : "+f"(b[m]));
            if (j + BB < 8) load(j + BB, v[(j / BB + 1) & 1]);
#pragma unroll
            for (int i = 0; i < BB; ++i) {
                const float2 p = __half22float2(*reinterpret_cast<const __half2*>(&w[j + i]));
                const float mp = BF16 ? fmaf(-128.f, p.x, p.y) : p.y;
                const float d = p.x * unpos((j + i) & 3);   // (exact: a power of two)
                const f32x2 m2 = pair2(mp, mp), d2 = pair2(d, d);
                f32x2 x2[MT / 2];
                if constexpr (MT == 2) x2[0] = *reinterpret_cast<const f32x2*>(sums + 8 * (j + i));
                else {
#pragma unroll
                    for (int m = 0; m < MT / 2; m += 2) {
                        const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(sums + 8 * (j + i) + 2 * m);
                        x2[m] = q.x; x2[m + 1] = q.y;
                    }
                }
#pragma unroll
                for (int m = 0; m < MT / 2; ++m) {   // (joined first: a block enters the running sum with two roundings at its size, not three)
                    const float* h = b + 2 * MT * i + 2 * m;
                    a[m] = fma2(d2, add2(pair2(h[0], h[1]), pair2(h[MT], h[MT + 1])), fma2(m2, x2[m], a[m]));
                }
            }
        }
#pragma unroll
        for (int m = 0; m < MT / 2; ++m) unpair2(a[m], acc[2 * m], acc[2 * m + 1]);
    }
}

}  // namespace aq
