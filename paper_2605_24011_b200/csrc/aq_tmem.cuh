// Instructions with the A operand in TMEM, and the stores that put it there: shared by the decode and the prefill kernels.
//
// A lane's slot of a fragment (aq_layout.cuh) is what tcgen05.st.16x128b takes from a lane: registers 4 f + r of instruction
// f = 2 j + h (block j, half h), register r = (row half) + 2 (pair).  The sixteen k of instruction f are then, in the order
// the instruction sees them, element 2 t + e of group c (0, 1):  k = 32 j + 8 t + 4 h + 2 c + e.  The other operand has to
// come in that order: operand_position.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

namespace aq {

// Where element k of a row lies in operand order: the same block of 32, position 16 h + 8 c + 2 t + e.
__host__ __device__ __forceinline__ constexpr int64_t operand_position(int64_t k) {
    return (k & ~(int64_t)31) + ((k >> 2) & 1) * 16 + ((k >> 1) & 1) * 8 + ((k >> 3) & 3) * 2 + (k & 1);
}
// Four consecutive elements from k (a multiple of 4): two pairs.
__device__ __forceinline__ void store_operand4(__half* row, int64_t k, const uint2& v) {
    uint32_t* p = reinterpret_cast<uint32_t*>(row + operand_position(k));
    p[0] = v.x;
    p[4] = v.y;
}
// Eight consecutive elements per lane, from k (a multiple of 8) where on; lanes 4 i .. 4 i + 3 hold a block of 32 and are on
// together; all lanes of the warp take part.  A lane's four pairs belong 16 bytes apart: the four lanes transpose them, and
// each stores 16 bytes in one piece (as 4-byte stores they were twice the number of partly written sectors).
__device__ __forceinline__ void store_operand8(__half* row, int64_t k, uint4 v, bool on) {
    const bool odd = threadIdx.x & 1, up = threadIdx.x & 2;
    uint32_t s0 = odd ? v.x : v.y, s1 = odd ? v.z : v.w;
    s0 = __shfl_xor_sync(0xffffffffu, s0, 1);
    s1 = __shfl_xor_sync(0xffffffffu, s1, 1);
    if (odd) { v.x = s0; v.z = s1; } else { v.y = s0; v.w = s1; }
    s0 = up ? v.x : v.z; s1 = up ? v.y : v.w;
    s0 = __shfl_xor_sync(0xffffffffu, s0, 2);
    s1 = __shfl_xor_sync(0xffffffffu, s1, 2);
    if (up) { v.x = s0; v.y = s1; } else { v.z = s0; v.w = s1; }
    if (on) *reinterpret_cast<uint4*>(row + k) = v;
}

__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
    return p != 0;
}
// A in TMEM, B in shared memory
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
// The same over a CTA pair: M = 256, each CTA holds its 128 rows of A in its TMEM and half of B in its shared memory
__device__ __forceinline__ void umma_f16_ts_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accum) : "memory");
}
__device__ __forceinline__ void tmem_st_16x128(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]),
          "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]),
          "r"(v[30]), "r"(v[31]) : "memory");
}
__device__ __forceinline__ void tmem_st_16x128(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
          "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

}  // namespace aq
