// Decode path for a whole program of linears (M = 1..8) in ONE persistent
// kernel launch (Section 4.3: the deployed forward pass dispatches every
// quantised matmul to a low-bit kernel; Appendix D: dequantise on the fly).
//
// Bound: HBM -- every packed byte of every matrix is read once per pass.  A
// 4096 x 4096 matrix is about a microsecond of HBM time, less than a kernel
// launch, so the pass runs as one cooperative grid of one CTA per SM:
//
//   * Work.  Consecutive ops that read the same input vector form a phase.
//     Every op's units (128 rows x 256 k) are dealt as contiguous runs to the
//     CTAs.  Inside a CTA five roles pass the units on (aq_decode_tc.cuh has the
//     arithmetic), so that none waits for another's latency:
//       - the feeder (one thread) keeps a ring of bulk copies (cp.async.bulk +
//         mbarrier, L2 evict-first) full;
//       - eight unpack warps turn codes into tensor-core operands in TMEM, in two
//         or five stages.  Neither depends on any activation: they run ahead
//         across op and phase boundaries, so a phase starts with its first units
//         waiting in TMEM;
//       - the issuer (one thread) starts a unit's tensor-core instructions;
//       - eight or twelve collect warps (ds_teams) form a phase's input, read the units'
//         sums back, apply scales and minima and add the rows up in memory;
//       - two record warps write the caller's copies of a phase's input.
//     Four warps that each did all of this in turn, step after step, needed 1404
//     us for a 7B-shaped pass of one token (software-pipelined: 1398); the roles
//     834, the mma.sync kernel before them 1044 (3.4 against 2.7 TB/s).
//   * Sums and dependencies.  A row's sum over a unit leaves its lane as ONE
//     64-bit red.add: the sum in 2^-24 fixed point in the upper 52 bits plus 1 in
//     the lower 12.  A row is complete when its count equals the number of
//     k-slabs of the matrix, so whoever needs a value polls the value
//     itself: no arrival counters, no fences, no release, and the result does
//     not depend on the order of the additions.  A CTA starts a phase as soon
//     as the elements IT reads are complete, not when the whole op is.
//   * Glue.  At the start of a phase each CTA forms, in shared memory, the
//     rounded input vector for the k-slabs its units touch (RMS scaling /
//     SiLU(g)*u / plain) with one round trip to L2.  Its share of the float32
//     buffer and of the rounded vector goes to the caller's workspace, where
//     every op's input and output stay readable.
//
// What bounds it now (7B shapes, one token): between two boundaries a unit takes
// 304 ns per SM, HBM's rate is 323; a boundary costs 3.3 us, of which the ring
// (160 KB per SM, 3.6 us of HBM) hides the weights' part.  With 8 tokens the collect
// warps set the pace: a team of four takes 1.7 us per unit, 0.7 to read the sums and
// apply the block scales and 1 for 1024 red.adds, and a boundary costs about 9 us, most
// of it the wait for the slowest CTA and the exchange of row norms.  Two teams, with A
// kept until the sums were read and one multiply-add per value, took 2306 us for a 7B-shaped
// pass, two teams with operand and sums released on their own 2278, three 2180.  Neither
// the L2 rate of the adds (204 ns per 1024 of them with every SM adding) nor the polls
// (pauses of 32 to 250 ns in them changed nothing) is the limit.  The order in which the
// compiler lays out the roles moves these figures by up to 8 %: measure after any change.
//
// Every wait is bounded: when one runs out the kernel raises a status word,
// gives copies in flight time to land and returns.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>
#include <mutex>
#include <numeric>
#include <type_traits>
#include <vector>

#include "aq_decode_rings.h"
#include "aq_decode_tc.cuh"
#include "aq_internal.h"

namespace aq {

typedef unsigned long long u64;

// Warps by role (a warp reaches the TMEM lanes of its quarter only: unpack and collect teams start at multiples of four).
constexpr int DS_UNPACK_WARPS = 8;          // two teams of four: one per half (128 k) of a unit
constexpr int DS_RECORD_WARPS = 2;
// Collect warps: teams of four that take the units in turn, two or three (ds_teams).  With three, registers are dealt to the roles
// by what they need (-Xptxas -v: 80 registers, 16 and 28 bytes spilled for binary16 and bfloat16; two teams 90 to 96 registers,
// none to 4 bytes spilled, with eight tokens 16 and 20).
template <int NTEAMS> struct DsRoles {
    static constexpr int TEAMS = NTEAMS, COLLECT_WARPS = 4 * TEAMS, CTHREADS = COLLECT_WARPS * 32;
    static constexpr int COLLECT0 = DS_UNPACK_WARPS, ISSUER = COLLECT0 + COLLECT_WARPS, FEEDER = ISSUER + 1, RECORD0 = FEEDER + 1;
    static constexpr int WARPS = RECORD0 + DS_RECORD_WARPS, THREADS = WARPS * 32;
    static constexpr bool SHARES = TEAMS == 3;      // registers per thread: 80 at the launch, then
    static constexpr int REGS_UNPACK = 56, REGS_COLLECT = 104, REGS_OTHER = 56;
    static_assert(!SHARES || DS_UNPACK_WARPS * REGS_UNPACK + COLLECT_WARPS * REGS_COLLECT + 4 * REGS_OTHER <= WARPS * 80, "the roles' registers fit");
    static_assert(!SHARES || (COLLECT0 % 4 == 0 && ISSUER % 4 == 0 && WARPS - ISSUER == 4), "no group of four has two shares");
};
constexpr int DS_MAX_COLLECT_WARPS = 12;
constexpr int DS_FRAGS = 8;                 // 16-row tiles of a unit
constexpr int DS_QUEUE = 16;                // units in flight at most
constexpr int DS_RING_BYTES = 160 * 1024;   // packed units in flight
constexpr int DS_MAX_SLOTS = 6;             // staged slabs per phase per CTA
constexpr int DS_XS_BYTES = DS_MAX_SLOTS * dt_slab_bytes(AQ_DECODE_MAX_M);
// A unit's operands and sums in TMEM, A of both halves and D of both halves, and what goes with it (descriptor, scales, the
// barrier that says they are there).  One token: five stages of both, refilled once the sums have been read.  Several tokens:
// reading the sums takes longer than anything else, so A (two stages) is refilled as soon as the instructions have read it (ds_late: where that pays)
// and D (two as well) is written again once the sums have been read (aq_decode_rings.h).
constexpr int DS_MAX_STAGES = 5;
template <int MT> struct DsStage {
    static constexpr int A_COLS = 2 * DtShape<MT>::A_COLS, D_COLS = 2 * DtShape<MT>::D_COLS;   // 64 + 32 / 128 + 128
    static constexpr bool SPLIT = MT > 1;
    static constexpr int A = SPLIT ? DS_A_STAGES : 5, D = SPLIT ? DS_D_STAGES : 5, META = SPLIT ? DS_META_SLOTS : 5;
    static_assert(A * A_COLS + D * D_COLS <= 512 && A <= DS_MAX_STAGES && D <= DS_MAX_STAGES && META <= DS_MAX_STAGES, "fits TMEM and the barriers");
    // first columns of stages (one token: a stage's sums lie behind its operand, one address serves both)
    __device__ static __forceinline__ uint32_t a_col(uint32_t s) { return s * (SPLIT ? A_COLS : A_COLS + D_COLS); }
    __device__ static __forceinline__ uint32_t d_col(uint32_t s) { return SPLIT ? A * A_COLS + s * D_COLS : a_col(s) + A_COLS; }
};
// A slot of a ring and how often the ring has gone round.
template <int N> struct DsRing {
    uint32_t at = 0, use = 0;
    __device__ __forceinline__ void next() { if (++at == N) { at = 0; ++use; } }
};
// Where the next unit lies: its A stage, D stage and what goes with it (one token: all the same).
template <int MT> struct DsPlace {
    DsRing<DsStage<MT>::A> ra;
    DsRing<DsStage<MT>::D> rd;
    DsRing<DsStage<MT>::META> rm;
    __device__ __forceinline__ const auto& a() const { return ra; }
    __device__ __forceinline__ const auto& d() const { return rd; }
    __device__ __forceinline__ const auto& m() const { return rm; }
    __device__ __forceinline__ void next() { ra.next(); rd.next(); rm.next(); }
};
template <> struct DsPlace<1> {
    DsRing<DsStage<1>::A> r;
    __device__ __forceinline__ const auto& a() const { return r; }
    __device__ __forceinline__ const auto& d() const { return r; }
    __device__ __forceinline__ const auto& m() const { return r; }
    __device__ __forceinline__ void next() { r.next(); }
};
constexpr int DS_MAX_PHASE_OPS = 8;
constexpr int DS_RMS_HOLD = 4;              // groups of four elements per thread kept in registers by the one-token RMS path
// Several tokens: up to this many elements (M K) every CTA reads the rows whole for the row norms, above it the norms come from
// shares.  Whole rows cost 8 M K bytes from the same lines of L2, shares one more trip through L2 and a wait for the slowest
// CTA.  Measured on passes of 18 and 8 blocks: K = 1024, M = 8 500 us whole, 595 us shares; K = 4096, M = 4 (16384) 425
// against 441; K = 4096, M = 8 (32768) 634 against 588.
constexpr int64_t DS_WHOLE_ROWS = 16384;
constexpr int DS_RECS = 4;                  // phase records held in shared memory
constexpr int DS_DESC_FIRST = 8;            // descriptor word 0: op inside the phase | the op's first k-slab << 3 ...
constexpr int DS_DESC_BITS_SHIFT = 8;       // ... | code width << 8 ...
constexpr int DS_DESC_PHASE_SHIFT = 12;     // ... and the phase from bit 12 on
constexpr uint32_t DS_DESC_END = 0xFFFFFFFFu;   // ... or: the stream is over
constexpr u64 DS_WAIT_NS_DEFAULT = 2000000000ull;   // every wait gives up after two seconds

// A packed sum: bits [12, 64) hold the value in units of 2^-24 (two's complement), bits [0, 12) the number of
// contributions added so far.
constexpr int DS_CNT_BITS = 12;
constexpr u64 DS_CNT_MASK = (1ull << DS_CNT_BITS) - 1;
constexpr int DS_MAX_CONTRIB = (1 << DS_CNT_BITS) - 1;
constexpr float DS_FIX_ONE = 16777216.f;            // 2^24
constexpr float DS_FIX_MAX = 134217600.f;           // just below 2^27: what the 52-bit field holds with room to add

__device__ int g_decode_status = 0;   // nonzero: a bounded wait ran out (1 = an input never completed, 2 = a copy)

struct DsOp {
    u64* dst;              // packed sums [M][N]
    const void* res;       // [M][N] added once (by the k-slab-0 units), or null: packed sums that are complete before the
                           // phase starts, or plain float32 when res_plain is set (the program input)
    int32_t N;             // true rows
    int32_t res_plain;
    u64 pad_;
};

struct DsPhase {
    const u64* src;        // packed [M][K], or null when the source is plain float32
    const u64* src2;       // second input of AQ_IN_SILU_MUL (packed), else null
    const float* src_f;    // plain float32 [M][K] source (the program input), used when src is null
    const float* src2_f;
    float* rec;            // float32 [M][K]: the caller's copy of src, written share by share (null: nothing to write)
    float* rec2;
    void* stage;           // [M][K] of the activation dtype: the rounded input, kept for the caller
    int32_t K;
    int32_t in_op;
    int32_t op_count;
    uint32_t expect;       // contributions that complete an element of src
    uint32_t expect2;
    int32_t pad_[1];
    u64* norm;             // [CTAs][M] (sum of squares over the CTA's share of the row | 1 << 32), zero before the
                           // pass; null: every CTA reads whole rows for the norm itself
    u64 pad2_;
    DsOp ops[DS_MAX_PHASE_OPS];
};
static_assert(sizeof(DsOp) == 32, "DsOp layout");
static_assert(sizeof(DsPhase) % 16 == 0, "a phase record is fetched with one bulk copy");

// What the feeder needs to know of an op, in the order of the program.
struct DsFeedOp {
    const uint8_t* frags;
    int32_t units_q;       // KP NT8 = units_q * (number of CTAs) + units_r (NT8: 128-row tiles)
    int32_t units_r_rot;   // units_r | rot << 16: CTA c takes the run of slot (c + rot) mod (number of CTAs)
    int32_t NT;            // 16-row tiles
    uint32_t word0;        // descriptor word 0 without the first-slab bit
    int32_t pad_[2];
};
static_assert(sizeof(DsFeedOp) == 32, "DsFeedOp layout");
// What one CTA needs to know of one phase besides the phase record: worked out on the host, since it depends on
// nothing but the shapes (a single thread doing this in the kernel sat on every phase's critical path).
struct DsCtaPhase {
    int32_t total;                          // units of the phase dealt to this CTA
    int32_t n_slots;                        // staged slabs
    int32_t slab_of_slot[DS_MAX_SLOTS];     // the pair-slabs staged for the phase, ascending
};
static_assert(sizeof(DsCtaPhase) == 32, "DsCtaPhase layout");

// A stretch of a buffer no phase reads: converted to float32 for the caller once the last phase is done.
struct DsTail {
    const u64* src;
    float* out;
    int32_t n;
    uint32_t expect;
    int32_t pad_[2];
};
static_assert(sizeof(DsTail) == 32, "DsTail layout");
// Elements per chunk: four groups of four per lane of a warp, whose readings go out together.  (With 2048 read one group after the
// other a launch ended 5 us later: an MLP of 4096 / 11008 and one token 30.7 us.)
constexpr int DS_TAIL_CHUNK = 512;

struct DsArgs {
    const DsPhase* phases;
    const DsFeedOp* feed_ops;         // n_ops entries and a spare one
    const int16_t* xoff;              // [op][CTA]: (slot of the CTA's first slab) - (that slab): slab P is staged in slot xoff + P
    const int32_t* unit_total;        // [CTA]: its units over all phases
    const DsTail* tails;
    const DsCtaPhase* ctab;           // [phase][CTA]
    u64 wait_ns;
    int n_phases;
    int n_ops;
    int n_tails;
    int M;
    int late;                         // several tokens: a unit is unpacked only when the sums of the last one in its stage have been read
    // the caller's rounded output: the tail chunks that convert [out_src, out_src + out_n) also write it (null: nobody does)
    void* out;
    const u64* out_src;
    int64_t out_n;
};

// ---- small PTX wrappers ---------------------------------------------------------
__device__ __forceinline__ uint32_t ds_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ds_mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void ds_mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void ds_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool ds_mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void ds_bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
        ::"r"(dst), "l"(src), "r"(bytes), "r"(bar), "l"(pol) : "memory");
}
__device__ __forceinline__ uint64_t ds_now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait on a shared-memory barrier; false when wait_ns passed (the status is raised) or another role gave up.
__device__ __forceinline__ bool ds_mbar_wait(uint32_t bar, uint32_t parity, u64 wait_ns, int* abort_flag) {
    if (ds_mbar_try(bar, parity)) return true;
    const uint64_t t0 = ds_now_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (ds_mbar_try(bar, parity)) return true;
        if (*reinterpret_cast<volatile int*>(abort_flag) != 0) return false;
        if (ds_now_ns() - t0 > wait_ns) {
            atomicCAS(&g_decode_status, 0, 2);
            *reinterpret_cast<volatile int*>(abort_flag) = 1;
            return false;
        }
    }
}
// The same by a whole warp, with one answer for all of it.
__device__ __forceinline__ bool ds_warp_wait(uint32_t bar, uint32_t parity, u64 wait_ns, int* abort_flag) {
    return __all_sync(0xffffffffu, ds_mbar_wait(bar, parity, wait_ns, abort_flag));
}
// Barrier among the collect warps only.
template <int THREADS>
__device__ __forceinline__ void ds_collect_sync() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }
// The same barrier, returning the OR of `flag` over all collect threads: every thread gets the same answer, so a
// decision to leave the phase loop is taken by all warps or by none (a flag read after a plain barrier could change
// between two threads' reads).
template <int THREADS>
__device__ __forceinline__ bool ds_collect_sync_or(int flag) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r) : "r"(flag), "n"(THREADS) : "memory");
    return r != 0;
}

// ---- packed sums ------------------------------------------------------------------
__device__ __forceinline__ u64 ds_pack(float v) {
    v = fminf(fmaxf(v, -DS_FIX_MAX), DS_FIX_MAX);
    return ((u64)__float2ll_rn(v * DS_FIX_ONE) << DS_CNT_BITS) + 1ull;
}
__device__ __forceinline__ float ds_unpack(u64 w) { return __ll2float_rn((long long)w >> DS_CNT_BITS) * (1.f / DS_FIX_ONE); }
__device__ __forceinline__ void ds_ld2(const u64* p, u64& a, u64& b) {
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ u64 ds_ld1(const u64* p) {
    u64 a;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
    return a;
}
__device__ __forceinline__ void ds_red_add(u64* p, u64 v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
struct DsQuad { u64 w[4]; };
__device__ __forceinline__ void ds_ld_quad(const u64* p, DsQuad& q) { ds_ld2(p, q.w[0], q.w[1]); ds_ld2(p + 2, q.w[2], q.w[3]); }
__device__ __forceinline__ bool ds_quad_ready(const DsQuad& q, uint32_t expect) {
    return (uint32_t)(q.w[0] & DS_CNT_MASK) == expect && (uint32_t)(q.w[1] & DS_CNT_MASK) == expect &&
           (uint32_t)(q.w[2] & DS_CNT_MASK) == expect && (uint32_t)(q.w[3] & DS_CNT_MASK) == expect;
}
__device__ __forceinline__ float4 ds_quad_value(const DsQuad& q) {
    return make_float4(ds_unpack(q.w[0]), ds_unpack(q.w[1]), ds_unpack(q.w[2]), ds_unpack(q.w[3]));
}
// Re-reads four packed sums until all are complete; false (status raised) when the wait runs out or the grid gave up.
__device__ __noinline__ bool ds_quad_wait(const u64* p, DsQuad& q, uint32_t expect, u64 wait_ns, int* abort_flag) {
    const uint64_t t0 = ds_now_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 16; ++i) {
            ds_ld_quad(p, q);
            if (ds_quad_ready(q, expect)) return true;
        }
        if (*reinterpret_cast<volatile int*>(&g_decode_status) != 0) { *abort_flag = 1; return false; }
        if (ds_now_ns() - t0 > wait_ns) { atomicCAS(&g_decode_status, 0, 1); *abort_flag = 1; return false; }
    }
}

// q holds a first reading of the four sums at p: true once they are complete (re-read as long as needed, into a
// copy of its own so that q itself can stay in registers).
__device__ __forceinline__ bool ds_quad_complete(const u64* p, DsQuad& q, uint32_t expect, u64 wait_ns, int* abort_flag) {
    if (ds_quad_ready(q, expect)) return true;
    DsQuad t;
    const bool ok = ds_quad_wait(p, t, expect, wait_ns, abort_flag);
    q = t;
    return ok;
}

// ---- glue arithmetic --------------------------------------------------------------
__device__ __forceinline__ float ds_silu_mul(float g, float u) { return g / (1.f + expf(-g)) * u; }

// Rounds four values to the activation dtype; *sum gets the sum of the rounded values.
template <bool BF16>
__device__ __forceinline__ uint2 ds_round4(const float4& v, float* sum) {
    uint2 r;
    if constexpr (BF16) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        r.x = *reinterpret_cast<uint32_t*>(&a); r.y = *reinterpret_cast<uint32_t*>(&b);
        const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
        *sum = (fa.x + fa.y) + (fb.x + fb.y);
    } else {
        __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
        r.x = *reinterpret_cast<uint32_t*>(&a); r.y = *reinterpret_cast<uint32_t*>(&b);
        const float2 fa = __half22float2(a), fb = __half22float2(b);
        *sum = (fa.x + fa.y) + (fb.x + fb.y);
    }
    return r;
}

// The four values of ds_round4's result.
template <bool BF16>
__device__ __forceinline__ float4 ds_values4(const uint2& r) {
    float2 a, b;
    if constexpr (BF16) { a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r.x)); b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&r.y)); }
    else { a = __half22float2(*reinterpret_cast<const __half2*>(&r.x)); b = __half22float2(*reinterpret_cast<const __half2*>(&r.y)); }
    return make_float4(a.x, a.y, b.x, b.y);
}

// ---- shared memory ------------------------------------------------------------------
struct DsShared {
    alignas(128) uint8_t ring[DS_RING_BYTES];
    alignas(128) uint8_t zlow[DT_ZERO_BYTES];   // (zeros below and above the slabs: see dt_issue)
    alignas(128) uint8_t xs[DS_XS_BYTES];       // staged input slabs
    alignas(128) uint8_t zhigh[DT_ZERO_BYTES];
    alignas(128) uint8_t dm[DS_MAX_STAGES][2 * DS_FRAGS][SCALE_BYTES];   // the staged units' scales and minima
    alignas(16) DsPhase rec[DS_RECS];       // phase records, fetched two phases ahead
    alignas(16) DsCtaPhase ctab[DS_RECS];   // this CTA's tables of the same phases
    alignas(16) uint4 desc[DS_QUEUE];       // units in the ring: (word 0, byte offset of the staged slab, 128-row tile, offset in the
                                            // ring | size of half a unit / 256 << 20)
    alignas(16) uint4 sdesc[DS_MAX_STAGES]; // the same of the units in TMEM
    alignas(8) uint64_t full[DS_QUEUE];     // the unit's copies have landed
    alignas(8) uint64_t empty[DS_QUEUE];    // the unpack warps have read it
    alignas(8) uint64_t stored[DS_MAX_STAGES];   // ... and stored its A operand
    alignas(8) uint64_t done[DS_MAX_STAGES];     // its tensor-core instructions have completed
    alignas(8) uint64_t taken[DS_MAX_STAGES];    // its sums have been read
    alignas(8) uint64_t rec_bar[DS_RECS];
    uint32_t qsize[DS_QUEUE];               // (the feeder's) ring bytes of the units in flight
    float red[AQ_DECODE_MAX_M][DS_MAX_COLLECT_WARPS];
    float scale[DS_RECS][AQ_DECODE_MAX_M];  // row scales of the phases (1 / rms)
    uint32_t tmem;
    int xphase;                             // phases whose input is staged
    int recorded[DS_RECORD_WARPS];          // phases whose caller's copies are written
    int abort_flag;
};
static_assert(sizeof(DsShared) <= 227 * 1024, "fits an SM");

// One packed red.add per token of the lane's row.  When `res` is given its value (complete, same shape as out) rides along.
template <int MT>
__device__ __forceinline__ void ds_commit(const float (&acc)[MT], u64* out, const void* res, bool res_plain, int row, int N, int M) {
    if (row >= N) return;
    if constexpr (MT > 2) {
        // (what a sum costs here, times 1024 per unit, is a third of the collect warps' instructions: the limits are looked at
        // once for all tokens; with two tokens that only delays the first, 18 expert blocks 269 -> 275 us)
        float mx = 0.f;
        bool clean = true;
#pragma unroll
        for (int m = 0; m < MT; ++m) { mx = fmaxf(mx, fabsf(acc[m])); clean = clean && acc[m] == acc[m]; }
        if (res == nullptr && clean && mx < DS_FIX_MAX) {
            u64* p = out + row;
#pragma unroll
            for (int m = 0; m < MT; ++m, p += N)
                if (m < M) ds_red_add(p, ((u64)__float2ll_rn(acc[m] * DS_FIX_ONE) << DS_CNT_BITS) + 1ull);
            return;
        }
    }
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        if (m >= M) break;
        const int64_t o = (int64_t)m * N + row;
        u64 w = ds_pack(acc[m]);
        if (res != nullptr) {
            if (res_plain) w += ds_pack(__ldcg(reinterpret_cast<const float*>(res) + o)) - 1ull;
            else w += ds_ld1(reinterpret_cast<const u64*>(res) + o) & ~DS_CNT_MASK;
        }
        ds_red_add(out + o, w);
    }
}

// ---- the roles ------------------------------------------------------------------------
// The CTA's units [a, b) of an op: slot s takes q + 1 units if s < r, else q.
__device__ __forceinline__ void ds_cta_run(int q, int r_rot, int& a, int& b) {
    const int r = r_rot & 0xFFFF, rot = r_rot >> 16;
    int s = (int)blockIdx.x + rot;
    if (s >= (int)gridDim.x) s -= (int)gridDim.x;
    a = q * s + min(s, r);
    b = a + q + (s < r ? 1 : 0);
}

// The feeder (one thread): every unit of the CTA, op by op, into the ring as soon as there is room.
__device__ __forceinline__ void ds_feed(DsShared& sh, const DsArgs& a) {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    uint32_t head = 0, room = DS_RING_BYTES;   // next byte of the ring, free bytes
    uint32_t nq = 0, tail = 0;                 // units copied, units known to have been read
    auto wait_tail = [&]() -> bool {
        const uint32_t e = tail % DS_QUEUE;
        if (!ds_mbar_wait(ds_smem(&sh.empty[e]), (tail / DS_QUEUE) & 1u, 2 * a.wait_ns, &sh.abort_flag)) return false;
        room += sh.qsize[e];
        ++tail;
        return true;
    };
    DsFeedOp next = a.feed_ops[0];             // (one op ahead: the latency hides behind an op's copies)
    int next_off = a.xoff[blockIdx.x];
    for (int o = 0; o < a.n_ops; ++o) {
        const DsFeedOp run = next;
        const int slab = next_off * dt_slab_bytes(a.M);
        next = a.feed_ops[o + 1];
        next_off = a.xoff[(size_t)(o + 1) * gridDim.x + blockIdx.x];
        int u0, u1;
        ds_cta_run(run.units_q, run.units_r_rot, u0, u1);
        const int fb = frag_bytes((int)(run.word0 >> DS_DESC_BITS_SHIFT) & 7), NT8 = (run.NT + DS_FRAGS - 1) / DS_FRAGS;
        int P = u0 / NT8, R = u0 - P * NT8;
        for (int u = u0; u < u1; ++u) {
            const uint32_t half = (uint32_t)(min(DS_FRAGS, run.NT - R * DS_FRAGS) * fb), need = 2 * half;
            const bool wrap = head + need > DS_RING_BYTES;             // (a unit lies in one piece)
            const uint32_t pad = wrap ? DS_RING_BYTES - head : 0u;
            while (room < need + pad || nq - tail == DS_QUEUE)
                if (!wait_tail()) return;
            if (wrap) head = 0;
            const uint32_t e = nq % DS_QUEUE, bar = ds_smem(&sh.full[e]);
            sh.qsize[e] = need + pad;
            // (ordered before the copies' arrival by the release of expect_tx)
            sh.desc[e] = make_uint4(run.word0 | (P == 0 ? (uint32_t)DS_DESC_FIRST : 0u), (uint32_t)(slab + P * dt_slab_bytes(a.M)), (uint32_t)R,
                                    head | ((half >> 8) << 20));
            ds_expect_tx(bar, need);
            const uint8_t* src = run.frags + frag_index(2 * P, R * DS_FRAGS, run.NT) * fb;
            ds_bulk_load(ds_smem(sh.ring) + head, src, half, bar, pol);
            ds_bulk_load(ds_smem(sh.ring) + head + half, src + (int64_t)run.NT * fb, half, bar, pol);
            room -= need + pad;
            head += need;
            ++nq;
            if (++R == NT8) { R = 0; ++P; }
        }
    }
    while (nq - tail >= DS_QUEUE)
        if (!wait_tail()) return;
    sh.desc[nq % DS_QUEUE] = make_uint4(DS_DESC_END, 0u, 0u, 0u);
    ds_mbar_arrive(ds_smem(&sh.full[nq % DS_QUEUE]));
}

// An unpack warp: its two fragments (rows 32 quarter .. + 31) of half `half` of every unit.
template <int MT, bool BF16>
__device__ __forceinline__ void ds_unpack_units(DsShared& sh, u64 wait_ns, uint32_t tmem, bool late, int half, int quarter, int lane) {
    using ST = DsStage<MT>;
    using SH = DtShape<MT>;
    const uint32_t released = ds_smem(late ? sh.taken : sh.done);   // several tokens: by which barriers
    DsPlace<MT> at;
    for (uint32_t n = 0;; ++n) {
        const uint32_t e = n % DS_QUEUE;
        if (!ds_warp_wait(ds_smem(&sh.full[e]), (n / DS_QUEUE) & 1u, wait_ns, &sh.abort_flag)) return;
        const uint4 d = sh.desc[e];
        if (d.x == DS_DESC_END) return;
        const int bits = (int)(d.x >> DS_DESC_BITS_SHIFT) & 7, fb = frag_bytes(bits);
        // (row tiles past the matrix's last one: whatever lies there; their rows are not written)
        const uint8_t* fr = sh.ring + (d.w & 0xFFFFFu) + (half ? (d.w >> 20) << 8 : 0u) + (uint32_t)(quarter * 2 * fb);
        const uint4 dm = *reinterpret_cast<const uint4*>(fr + (lane >> 4) * fb + (lane & 15) * 16);
        const uint32_t ta = tmem + ST::a_col(at.a().at) + (uint32_t)(half * SH::A_COLS) + ((uint32_t)(quarter * 32) << 16);
        // the stage is free once its last unit's instructions have completed (one token, and late: and its sums have been read)
        auto stage_free = [&]() {
            if (at.a().use == 0) return true;
            if constexpr (!ST::SPLIT) return ds_warp_wait(ds_smem(&sh.taken[at.a().at]), (at.a().use - 1) & 1u, wait_ns, &sh.abort_flag);
            const uint32_t before = n - ST::A;   // the unit that had the stage
            return ds_warp_wait(released + 8 * (before % ST::D), (before / ST::D) & 1u, wait_ns, &sh.abort_flag);
        };
        if constexpr (MT == 1) {
            uint32_t va[16], vb[16];
            if (bits == 2) dt_unpack2<2>(fr, lane, va, vb);
            else if (bits == 3) dt_unpack2<3>(fr, lane, va, vb);
            else dt_unpack2<4>(fr, lane, va, vb);
            if (!stage_free()) return;
            tc_fence_after();
            tmem_st_16x128(ta, va);
            tmem_st_16x128(ta + (16u << 16), vb);
        } else {
            // (the second fragment's words are loaded before the wait: what follows it delays the stage)
            auto both = [&](auto width) -> bool {
                constexpr int BITS = decltype(width)::value;
                LaneCodes<BITS> la, lb;
                load_lane_codes<BITS>(la, fr, lane);
                load_lane_codes<BITS>(lb, fr + fb, lane);
                uint32_t v[32];
                dt_unpack<BITS, BF16>(la, v);
                if (!stage_free()) return false;
                tc_fence_after();
                tmem_st_16x128(ta, v);
                dt_unpack<BITS, BF16>(lb, v);
                tmem_st_16x128(ta + (16u << 16), v);
                return true;
            };
            const bool ok = bits == 2 ? both(std::integral_constant<int, 2>()) : bits == 3 ? both(std::integral_constant<int, 3>()) : both(std::integral_constant<int, 4>());
            if (!ok) return;
        }
        *reinterpret_cast<uint4*>(&sh.dm[at.m().at][half * DS_FRAGS + quarter * 2 + (lane >> 4)][(lane & 15) * 16]) = dm;
        if (half == 0 && quarter == 0 && lane == 0) sh.sdesc[at.m().at] = d;
        tmem_st_wait();          // (everything read from the ring has been used: the slot may be refilled)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
            ds_mbar_arrive(ds_smem(&sh.empty[e]));
            ds_mbar_arrive(ds_smem(&sh.stored[at.m().at]));
        }
        at.next();
    }
}

// Waits until *count exceeds `value`; returns the count (not above `value`: gave up).  One answer for the whole warp.
__device__ __forceinline__ int ds_wait_count(const int* count, int value, u64 wait_ns, int* abort_flag) {
    const uint32_t addr = ds_smem(count);
    const uint64_t t0 = ds_now_ns();
    for (;;) {
        int v = 0;
#pragma unroll 1
        for (int i = 0; i < 256; ++i) {
            asm volatile("ld.acquire.cta.shared.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
            v = __shfl_sync(0xffffffffu, v, 0);
            if (v > value) return v;
        }
        const bool stop = *reinterpret_cast<volatile int*>(abort_flag) != 0 || ds_now_ns() - t0 > wait_ns;
        if (__any_sync(0xffffffffu, stop)) {
            if (*reinterpret_cast<volatile int*>(abort_flag) == 0) { atomicCAS(&g_decode_status, 0, 2); *reinterpret_cast<volatile int*>(abort_flag) = 1; }
            return v;
        }
    }
}

// The issuer (one warp, one elected thread): a unit's instructions once its A operand and the phase's input are there.
template <int MT, bool BF16>
__device__ __forceinline__ void ds_issue_units(DsShared& sh, const DsArgs& a, uint32_t tmem) {
    using ST = DsStage<MT>;
    DsPlace<MT> at;
    int ready = 0;   // phases whose input is staged
    const uint32_t zlow = ds_smem(sh.zlow), zhigh = ds_smem(sh.zhigh), xs = ds_smem(sh.xs);
    for (int left = a.unit_total[blockIdx.x]; left > 0; --left) {
        if (!ds_warp_wait(ds_smem(&sh.stored[at.m().at]), at.m().use & 1u, 2 * a.wait_ns, &sh.abort_flag)) return;
        if (ST::SPLIT && at.d().use > 0 && !ds_warp_wait(ds_smem(&sh.taken[at.d().at]), (at.d().use - 1) & 1u, 2 * a.wait_ns, &sh.abort_flag)) return;
        const uint2 d = *reinterpret_cast<const uint2*>(&sh.sdesc[at.m().at]);
        const int ph = (int)(d.x >> DS_DESC_PHASE_SHIFT);
        if (ready <= ph) {
            ready = ds_wait_count(&sh.xphase, ph, 2 * a.wait_ns, &sh.abort_flag);
            if (ready <= ph) return;
        }
        const uint32_t x = __shfl_sync(0xffffffffu, xs + d.y, 0);
        const uint32_t ta = __shfl_sync(0xffffffffu, tmem + ST::a_col(at.a().at), 0);
        uint32_t td = ta + ST::A_COLS;
        if constexpr (ST::SPLIT) td = __shfl_sync(0xffffffffu, tmem + ST::d_col(at.d().at), 0);
        tc_fence_after();
        if (elect_one()) {
            dt_issue<MT, BF16>(ta, td, x, zlow, zhigh);
            umma_commit(ds_smem(&sh.done[at.d().at]));
        }
        __syncwarp();
        at.next();
    }
}

// How the waits for other CTAs' sums end: a counter of rounds, the time of the first late one.
struct DsPatience {
    uint32_t spins = 0;
    uint64_t t0 = 0;
    // after a round of readings that found something incomplete: true when the wait has to end
    __device__ __forceinline__ bool over(DsShared& sh, u64 wait_ns) {
        if ((++spins & 7u) != 0) return false;
        if (*reinterpret_cast<volatile int*>(&g_decode_status) != 0) { sh.abort_flag = 1; return true; }
        const uint64_t t = ds_now_ns();
        if (t0 == 0) t0 = t;
        if (t - t0 > wait_ns) { atomicCAS(&g_decode_status, 0, 1); sh.abort_flag = 1; return true; }
        return false;
    }
};
// Four consecutive source elements at offset o, complete; zeros after a failed wait.
__device__ __forceinline__ float4 ds_source4(DsShared& sh, const u64* p, const float* pf, uint32_t expect, int64_t o, u64 wait_ns, DsPatience& pat) {
    if (p == nullptr) return __ldcg(reinterpret_cast<const float4*>(pf + o));
    DsQuad q;
    for (;;) {
        ds_ld_quad(p + o, q);
        if (ds_quad_ready(q, expect)) return ds_quad_value(q);
        if (pat.over(sh, wait_ns)) return make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// A record warp: this CTA's share of the caller's copies (the float32 source buffers and the rounded input of every
// phase), written while the phase's units are at work.
template <bool BF16>
__device__ __forceinline__ void ds_record(DsShared& sh, const DsArgs& a, int rw, int lane) {
    for (int ph = 0; ph < a.n_phases; ++ph) {
        const int pb = ph % DS_RECS;
        if (!ds_warp_wait(ds_smem(&sh.rec_bar[pb]), (uint32_t)(ph / DS_RECS) & 1u, 2 * a.wait_ns, &sh.abort_flag)) return;
        if (ds_wait_count(&sh.xphase, ph, 2 * a.wait_ns, &sh.abort_flag) <= ph) return;   // (the row scales are there then)
        const DsPhase& P = sh.rec[pb];
        const int q4 = P.K >> 2;                                  // groups of 4 elements per token
        const int g0 = (int)(((int64_t)q4 * blockIdx.x) / gridDim.x), share = (int)(((int64_t)q4 * (blockIdx.x + 1)) / gridDim.x) - g0;
        const bool two = (P.in_op == AQ_IN_SILU_MUL);
        DsPatience pat;
        for (int it = rw * 32 + lane; it < share * a.M; it += DS_RECORD_WARPS * 32) {
            const int m = it / share;
            const int64_t o = (int64_t)m * P.K + 4 * (int64_t)(g0 + it - m * share);
            float4 v = ds_source4(sh, P.src, P.src_f, P.expect, o, a.wait_ns, pat);
            if (P.rec) *reinterpret_cast<float4*>(P.rec + o) = v;
            if (two) {
                const float4 t = ds_source4(sh, P.src2, P.src2_f, P.expect2, o, a.wait_ns, pat);
                if (P.rec2) *reinterpret_cast<float4*>(P.rec2 + o) = t;
                v = make_float4(ds_silu_mul(v.x, t.x), ds_silu_mul(v.y, t.y), ds_silu_mul(v.z, t.z), ds_silu_mul(v.w, t.w));
            } else {
                const float sc = (P.in_op == AQ_IN_RMSNORM) ? sh.scale[pb][m] : 1.f;
                v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
            }
            float sum;
            *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(P.stage) + o) = ds_round4<BF16>(v, &sum);
        }
        __syncwarp();
        if (lane == 0) asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(ds_smem(&sh.recorded[rw])), "r"(ph + 1) : "memory");
    }
}

// Asks for a phase's record and this CTA's tables for it, on one barrier.
__device__ __forceinline__ void ds_fetch_record(DsShared& sh, const DsArgs& a, int q) {
    const uint32_t bar = ds_smem(&sh.rec_bar[q % DS_RECS]);
    uint64_t pol_keep;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
    ds_expect_tx(bar, (uint32_t)(sizeof(DsPhase) + sizeof(DsCtaPhase)));
    ds_bulk_load(ds_smem(&sh.rec[q % DS_RECS]), a.phases + q, (uint32_t)sizeof(DsPhase), bar, pol_keep);
    ds_bulk_load(ds_smem(&sh.ctab[q % DS_RECS]), a.ctab + (size_t)q * gridDim.x + blockIdx.x, (uint32_t)sizeof(DsCtaPhase), bar, pol_keep);
}

// ---- the kernel ---------------------------------------------------------------------
template <int MT, int TEAMS, bool BF16>
__global__ void __launch_bounds__(DsRoles<TEAMS>::THREADS, 1) decode_stack_kernel(const DsArgs a) {
    using ST = DsStage<MT>;
    using RO = DsRoles<TEAMS>;
    static_assert(!ST::SPLIT || ds_rings_hold(ST::A, ST::D, ST::META, TEAMS), "a slot is written again only when its last unit is through with it");
    extern __shared__ __align__(128) uint8_t ds_smem_raw[];
    DsShared& sh = *reinterpret_cast<DsShared*>(ds_smem_raw);
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int quarter = warp & 3;   // (a warp reaches the TMEM lanes of its quarter only)
    const int M = a.M;
    const u64 wait_ns = a.wait_ns;
    pdl_launch_dependents();   // (an attention step that follows may read its cache on the SMs this launch leaves first)

    // Two teams: a thread per barrier, and the first phases' records are asked for by the thread that has set up theirs.
    // (One thread for all of them, and the records after the CTA had met: an MLP of 2048 / 8192 took 4 to 9 % longer.  With
    // registers dealt by role the former costs 40 bytes of spills and 3 % of a 7B-shaped pass.)
    if constexpr (!RO::SHARES) {
        if (threadIdx.x < DS_QUEUE) {
            ds_mbar_init(ds_smem(&sh.full[threadIdx.x]), 1);
            ds_mbar_init(ds_smem(&sh.empty[threadIdx.x]), DS_UNPACK_WARPS);
        } else if (threadIdx.x >= 32 && threadIdx.x < 32 + DS_MAX_STAGES) {
            const int i = (int)threadIdx.x - 32;
            ds_mbar_init(ds_smem(&sh.stored[i]), DS_UNPACK_WARPS);
            ds_mbar_init(ds_smem(&sh.done[i]), 1);
            ds_mbar_init(ds_smem(&sh.taken[i]), 4);
        }
    }
    if (threadIdx.x == RO::COLLECT0 * 32) {
        sh.abort_flag = 0;
        sh.xphase = 0;
#pragma unroll
        for (int i = 0; i < DS_RECORD_WARPS; ++i) sh.recorded[i] = 0;
#pragma unroll 1
        for (int i = 0; i < DS_RECS; ++i) ds_mbar_init(ds_smem(&sh.rec_bar[i]), 1);
        if constexpr (!RO::SHARES) {
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_async_smem();
            if (a.n_phases > 0) ds_fetch_record(sh, a, 0);
            if (a.n_phases > 1) ds_fetch_record(sh, a, 1);
        } else {
#pragma unroll 1
            for (int i = 0; i < DS_QUEUE; ++i) {
                ds_mbar_init(ds_smem(&sh.full[i]), 1);
                ds_mbar_init(ds_smem(&sh.empty[i]), DS_UNPACK_WARPS);
            }
#pragma unroll 1
            for (int i = 0; i < DS_MAX_STAGES; ++i) {
                ds_mbar_init(ds_smem(&sh.stored[i]), DS_UNPACK_WARPS);
                ds_mbar_init(ds_smem(&sh.done[i]), 1);
                ds_mbar_init(ds_smem(&sh.taken[i]), 4);
            }
        }
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ds_smem(&sh.tmem)), "n"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the slabs keep zeros everywhere but in the elements the stagers rewrite every phase (rows of absent tokens; one
    // token: every row but the first)
    for (int i = threadIdx.x; i < (DS_XS_BYTES + 2 * DT_ZERO_BYTES) / 16; i += RO::THREADS)
        reinterpret_cast<uint4*>(sh.zlow)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem;

    // (The issuer, the feeder and the record warps are one group of four: setmaxnreg is for a whole group, so it stands in front of
    // the roles.  With the roles in a branch of their own behind it a 7B-shaped pass of 8 tokens took 2364 us instead of 2190.)
    if constexpr (RO::SHARES) {
        if (warp >= RO::ISSUER) { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(RO::REGS_OTHER)); }
    }
    if (warp < DS_UNPACK_WARPS) {
        if constexpr (RO::SHARES) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(RO::REGS_UNPACK));
        ds_unpack_units<MT, BF16>(sh, wait_ns, tmem, a.late != 0, warp >> 2, quarter, lane);
    } else if (warp == RO::ISSUER) {
        ds_issue_units<MT, BF16>(sh, a, tmem);
    } else if (warp == RO::FEEDER) {
        if (lane == 0) ds_feed(sh, a);
        __syncwarp();
    } else if (warp >= RO::RECORD0) {
        ds_record<BF16>(sh, a, warp - RO::RECORD0, lane);
    } else {
    if constexpr (RO::SHARES) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(RO::REGS_COLLECT));
    // ================= collect warps =================
    const int ctid = (int)threadIdx.x - RO::COLLECT0 * 32, cwarp = warp - RO::COLLECT0;
    if (RO::SHARES && ctid == 0) {
        if (a.n_phases > 0) ds_fetch_record(sh, a, 0);
        if (a.n_phases > 1) ds_fetch_record(sh, a, 1);
    }
    DsPlace<MT> at;                    // of the next unit
    uint32_t turn = 0;                 // the team whose unit that is

#pragma unroll 1
    for (int ph = 0; ph < a.n_phases; ++ph) {
        const int pb = ph % DS_RECS;
        const DsPhase& P = sh.rec[pb];
        const DsCtaPhase& C = sh.ctab[pb];
        // -- the phase's descriptors (fetched two phases ahead) --
        ds_mbar_wait(ds_smem(&sh.rec_bar[pb]), (uint32_t)(ph / DS_RECS) & 1u, wait_ns, &sh.abort_flag);
        if (cwarp == 0 && ph + 2 < a.n_phases) {   // slot of phase ph - 2: the collect warps are through with it, and the record warps?
#pragma unroll
            for (int i = 0; i < DS_RECORD_WARPS; ++i)
                if (ph >= 2) ds_wait_count(&sh.recorded[i], ph - 2, wait_ns, &sh.abort_flag);
            if (lane == 0) ds_fetch_record(sh, a, ph + 2);
        }
        // every warp is through with phase ph - 1: the staged slabs are free
        if (ds_collect_sync_or<RO::CTHREADS>(*reinterpret_cast<volatile int*>(&sh.abort_flag))) break;

        // -- form the rounded input vector for the slabs this CTA reads --
        {
            const int n_slots = C.n_slots;
            const int q4 = P.K >> 2;                                  // groups of 4 elements per token
            const uint32_t expect = P.expect, expect2 = P.expect2;
            DsPatience pat;
            // stores group i4 (elements 4 i4 ..) of token m into slab copy `sl`; whole warps call this together
            auto place = [&](uint8_t* sl, int m, int i4, float4 v) {
                float sum;
                const uint2 r = ds_round4<BF16>(v, &sum);   // v is zero past the end of the row: padding stages zeros
                const int kl = (i4 * 4) & 255;
                // block sums (and, for one token, the largest magnitude): 8 consecutive groups = 8 consecutive lanes
                sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                sum += __shfl_xor_sync(0xffffffffu, sum, 4);
                if constexpr (MT == 1) {
                    const float4 f = ds_values4<BF16>(r);
                    float mx = fmaxf(fmaxf(fabsf(f.x), fabsf(f.y)), fmaxf(fabsf(f.z), fabsf(f.w)));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
                    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
                    const uint32_t sc = dt_fix_scale(mx);
                    dt_stage4_fix(sl, kl, f, sc);
                    if ((lane & 7) == 0) reinterpret_cast<float2*>(sl + DT_SUMS<1>)[kl >> 5] = make_float2(sum, dt_fix_step(sc, sum));
                } else {
                    dt_stage4(sl, m, kl, r);
                    if ((lane & 7) == 0) reinterpret_cast<float*>(sl + DT_SUMS<MT>)[(kl >> 5) * 8 + m] = sum;
                }
            };
            if (P.in_op == AQ_IN_RMSNORM && MT == 1 && q4 <= DS_RMS_HOLD * RO::CTHREADS) {
                // one token, row held in registers: one trip to L2 once the row is complete (all of a thread's readings
                // go out together and are repeated together until every one of them is complete)
                float4 v[DS_RMS_HOLD];
                int slabs[DS_MAX_SLOTS];
#pragma unroll
                for (int x = 0; x < DS_MAX_SLOTS; ++x) slabs[x] = C.slab_of_slot[x];
                if (P.src != nullptr) {
                    DsQuad q[DS_RMS_HOLD];
                    for (;;) {
                        bool ready = true;
#pragma unroll
                        for (int n = 0; n < DS_RMS_HOLD; ++n) {
                            const int i4 = ctid + n * RO::CTHREADS;
                            if (i4 < q4) ds_ld_quad(P.src + 4 * (int64_t)i4, q[n]);
                        }
#pragma unroll
                        for (int n = 0; n < DS_RMS_HOLD; ++n) {
                            const int i4 = ctid + n * RO::CTHREADS;
                            if (i4 < q4) ready = ready && ds_quad_ready(q[n], expect);
                        }
                        if (ready || pat.over(sh, wait_ns)) break;
                    }
                    const bool failed = *reinterpret_cast<volatile int*>(&sh.abort_flag) != 0;
#pragma unroll
                    for (int n = 0; n < DS_RMS_HOLD; ++n) {
                        const int i4 = ctid + n * RO::CTHREADS;
                        v[n] = (i4 < q4 && !failed) ? ds_quad_value(q[n]) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                } else {
#pragma unroll
                    for (int n = 0; n < DS_RMS_HOLD; ++n) {
                        const int i4 = ctid + n * RO::CTHREADS;
                        v[n] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (i4 < q4) v[n] = __ldcg(reinterpret_cast<const float4*>(P.src_f) + i4);
                    }
                }
                __syncwarp();
                float ss = 0.f;
#pragma unroll
                for (int n = 0; n < DS_RMS_HOLD; ++n) {
                    ss = fmaf(v[n].x, v[n].x, ss); ss = fmaf(v[n].y, v[n].y, ss);
                    ss = fmaf(v[n].z, v[n].z, ss); ss = fmaf(v[n].w, v[n].w, ss);
                }
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
                if (lane == 0) sh.red[0][cwarp] = ss;
                ds_collect_sync<RO::CTHREADS>();
                float tot = 0.f;
#pragma unroll
                for (int w = 0; w < RO::COLLECT_WARPS; ++w) tot += sh.red[0][w];
                const float scale = rsqrtf(tot / (float)P.K + 1e-6f);
                if (ctid == 0) sh.scale[pb][0] = scale;
#pragma unroll
                for (int n = 0; n < DS_RMS_HOLD; ++n) {
                    const int i4 = ctid + n * RO::CTHREADS;
                    if (n * RO::CTHREADS < q4) {   // the same for every thread: warps stay whole
                        const int slab = i4 >> 6;   // (a warp's 32 groups are half a slab)
                        int sl = -1;
#pragma unroll
                        for (int x = 0; x < DS_MAX_SLOTS; ++x) sl = (x < n_slots && slabs[x] == slab) ? x : sl;
                        if (sl >= 0)
                            place(sh.xs + (size_t)sl * dt_slab_bytes(MT), 0, i4, make_float4(v[n].x * scale, v[n].y * scale, v[n].z * scale, v[n].w * scale));
                    }
                }
            } else {
                bool normed = false;
                if constexpr (MT > 1) {
                if (P.in_op == AQ_IN_RMSNORM && P.norm != nullptr) {
                    // Row norms from shares, a warp per token row: it sums the squares of this CTA's share of the row,
                    // publishes the sum as a (float | 1 << 32) word and gathers every CTA's word; all sums run in a fixed
                    // order, so every CTA gets the same norms.
                    if (cwarp < M) {
                        const int g0 = (int)(((int64_t)q4 * blockIdx.x) / gridDim.x), g1 = (int)(((int64_t)q4 * (blockIdx.x + 1)) / gridDim.x);
                        float ss = 0.f;
                        for (int g = g0 + lane; g < g1; g += 32) {
                            const float4 v = ds_source4(sh, P.src, P.src_f, expect, (int64_t)cwarp * P.K + 4 * (int64_t)g, wait_ns, pat);
                            ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss); ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss);
                        }
                        __syncwarp();
#pragma unroll
                        for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
                        u64* row = P.norm + (size_t)cwarp * AQ_NORM_MAX_CTAS;
                        if (lane == 0) {
                            const u64 w = (u64)__float_as_uint(ss) | (1ull << 32);
                            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(row + blockIdx.x), "l"(w) : "memory");
                        }
                        constexpr int NW = AQ_NORM_MAX_CTAS / 32;
                        u64 w[NW];
                        for (;;) {
                            bool ready = true;
#pragma unroll
                            for (int i = 0; i < NW; ++i) { w[i] = 1ull << 32; if (lane + 32 * i < (int)gridDim.x) w[i] = ds_ld1(row + lane + 32 * i); }
#pragma unroll
                            for (int i = 0; i < NW; ++i) ready = ready && (w[i] >> 32) != 0;
                            if (ready || pat.over(sh, wait_ns)) break;
                        }
                        __syncwarp();
                        float tot = 0.f;
#pragma unroll
                        for (int i = 0; i < NW; ++i) tot += __uint_as_float((uint32_t)w[i]);
#pragma unroll
                        for (int d = 16; d > 0; d >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, d);
                        if (lane == 0) sh.scale[pb][cwarp] = rsqrtf(tot / (float)P.K + 1e-6f);
                    }
                    ds_collect_sync<RO::CTHREADS>();
                    normed = true;
                }
                }
                if (P.in_op == AQ_IN_RMSNORM && !normed) {
                    if constexpr (MT < 4) {
                        for (int m = 0; m < M; ++m) {
                            float ss = 0.f;
                            for (int i = ctid; i < q4; i += RO::CTHREADS) {
                                const float4 v = ds_source4(sh, P.src, P.src_f, expect, (int64_t)m * P.K + 4 * (int64_t)i, wait_ns, pat);
                                ss = fmaf(v.x, v.x, ss); ss = fmaf(v.y, v.y, ss); ss = fmaf(v.z, v.z, ss); ss = fmaf(v.w, v.w, ss);
                            }
                            __syncwarp();
#pragma unroll
                            for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
                            if (lane == 0) sh.red[m][cwarp] = ss;
                        }
                    } else {
                        // two tokens at a time: both readings go out together and are repeated together until complete
                        for (int m = 0; m < M; m += 2) {
                            float ss[2] = {0.f, 0.f};
                            const bool second = m + 1 < M;
                            for (int i = ctid; i < q4; i += RO::CTHREADS) {
                                const int64_t o = (int64_t)m * P.K + 4 * (int64_t)i;
                                float4 v = make_float4(0.f, 0.f, 0.f, 0.f), u = v;
                                if (P.src == nullptr) {
                                    v = __ldcg(reinterpret_cast<const float4*>(P.src_f + o));
                                    if (second) u = __ldcg(reinterpret_cast<const float4*>(P.src_f + o + P.K));
                                } else {
                                    DsQuad qa, qb;
                                    for (;;) {
                                        ds_ld_quad(P.src + o, qa);
                                        if (second) ds_ld_quad(P.src + o + P.K, qb);
                                        const bool ready = ds_quad_ready(qa, expect) && (!second || ds_quad_ready(qb, expect));
                                        if (ready || pat.over(sh, wait_ns)) break;
                                    }
                                    v = ds_quad_value(qa);
                                    if (second) u = ds_quad_value(qb);
                                }
                                ss[0] = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, ss[0]))));
                                ss[1] = fmaf(u.w, u.w, fmaf(u.z, u.z, fmaf(u.y, u.y, fmaf(u.x, u.x, ss[1]))));
                            }
                            __syncwarp();
#pragma unroll
                            for (int x = 0; x < 2; ++x) {
#pragma unroll
                                for (int d = 16; d > 0; d >>= 1) ss[x] += __shfl_xor_sync(0xffffffffu, ss[x], d);
                                if (lane == 0 && m + x < M) sh.red[m + x][cwarp] = ss[x];
                            }
                        }
                    }
                    ds_collect_sync<RO::CTHREADS>();
                    if (ctid < M) {
                        float tot = 0.f;
#pragma unroll
                        for (int w = 0; w < RO::COLLECT_WARPS; ++w) tot += sh.red[ctid][w];
                        sh.scale[pb][ctid] = rsqrtf(tot / (float)P.K + 1e-6f);
                    }
                    ds_collect_sync<RO::CTHREADS>();
                }
                // half a slab of one token (32 groups) per warp and item, NB items in flight
                constexpr int NB = MT == 1 ? 1 : 2;
                const int n_items = 2 * n_slots * M;
                const uint32_t by_m = (65536u + (uint32_t)M - 1) / (uint32_t)M;   // (v * by_m) >> 16 = v / M for v < 64
                const bool two = (P.in_op == AQ_IN_SILU_MUL), rms = (P.in_op == AQ_IN_RMSNORM);
                for (int it0 = cwarp; it0 < n_items; it0 += NB * RO::COLLECT_WARPS) {
                    int slot[NB], m[NB], i4[NB];
                    bool on[NB];
#pragma unroll
                    for (int n = 0; n < NB; ++n) {
                        const int it = it0 + n * RO::COLLECT_WARPS, v = it >> 1;
                        slot[n] = (int)(((uint32_t)v * by_m) >> 16);
                        m[n] = v - slot[n] * M;
                        i4[n] = 0; on[n] = false;
                        if (it < n_items) {
                            i4[n] = C.slab_of_slot[slot[n]] * 64 + (it & 1) * 32 + lane;
                            on[n] = i4[n] < q4;
                        }
                    }
                    // all readings go out together and are repeated together until complete
                    float4 s[NB], t[NB];
                    DsQuad qa[NB], qb[NB];
                    bool ready;
                    for (;;) {
                        ready = true;
#pragma unroll
                        for (int n = 0; n < NB; ++n) {
                            const int64_t o = (int64_t)m[n] * P.K + 4 * (int64_t)i4[n];
                            if (on[n]) {
                                if (P.src) ds_ld_quad(P.src + o, qa[n]);
                                else s[n] = __ldcg(reinterpret_cast<const float4*>(P.src_f + o));
                                if (two) {
                                    if (P.src2) ds_ld_quad(P.src2 + o, qb[n]);
                                    else t[n] = __ldcg(reinterpret_cast<const float4*>(P.src2_f + o));
                                }
                            }
                        }
#pragma unroll
                        for (int n = 0; n < NB; ++n) {
                            if (on[n] && P.src) ready = ready && ds_quad_ready(qa[n], expect);
                            if (on[n] && two && P.src2) ready = ready && ds_quad_ready(qb[n], expect2);
                        }
                        if (ready || pat.over(sh, wait_ns)) break;
                    }
                    __syncwarp();
#pragma unroll
                    for (int n = 0; n < NB; ++n) {
                        if (it0 + n * RO::COLLECT_WARPS >= n_items) break;
                        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (on[n] && ready) {
                            v = P.src ? ds_quad_value(qa[n]) : s[n];
                            if (two) {
                                const float4 u = P.src2 ? ds_quad_value(qb[n]) : t[n];
                                v = make_float4(ds_silu_mul(v.x, u.x), ds_silu_mul(v.y, u.y), ds_silu_mul(v.z, u.z), ds_silu_mul(v.w, u.w));
                            } else if (rms) {
                                const float sc = sh.scale[pb][m[n]];
                                v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
                            }
                        }
                        __syncwarp();
                        place(sh.xs + (size_t)slot[n] * dt_slab_bytes(MT), m[n], i4[n], v);
                    }
                }
            }
        }
        fence_async_smem();   // (the tensor core reads the slabs through the asynchronous proxy)
        if (ds_collect_sync_or<RO::CTHREADS>(*reinterpret_cast<volatile int*>(&sh.abort_flag))) break;
        if (ctid == 0) asm volatile("st.release.cta.shared.s32 [%0], %1;" ::"r"(ds_smem(&sh.xphase)), "r"(ph + 1) : "memory");

        // -- the sums of the phase's units, the teams taking turns --
        const int total = C.total;
        bool ok = true;
#pragma unroll 1
        for (int i = 0; i < total && ok; ++i) {
            if (turn == (uint32_t)(cwarp >> 2)) {
                ok = ds_warp_wait(ds_smem(&sh.stored[at.m().at]), at.m().use & 1u, wait_ns, &sh.abort_flag) &&
                     ds_warp_wait(ds_smem(&sh.done[at.d().at]), at.d().use & 1u, wait_ns, &sh.abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint4 d = sh.sdesc[at.m().at];
                const int bits = (int)(d.x >> DS_DESC_BITS_SHIFT) & 7;
                const float* sums = reinterpret_cast<const float*>(sh.xs + d.y + DT_SUMS<MT>);
                const uint8_t* dmp = &sh.dm[at.m().at][quarter * 2 + (lane >> 4)][(lane & 15) * 16];
                const uint4 dm0 = *reinterpret_cast<const uint4*>(dmp), dm1 = *reinterpret_cast<const uint4*>(dmp + DS_FRAGS * SCALE_BYTES);
                const uint32_t td = tmem + ST::d_col(at.d().at) + ((uint32_t)(quarter * 32) << 16);
                float acc[MT];
#pragma unroll
                for (int m = 0; m < MT; ++m) acc[m] = 0.f;
                if (bits == 2) dt_collect<2, MT, BF16>(td, dm0, dm1, sums, acc);
                else if (bits == 3) dt_collect<3, MT, BF16>(td, dm0, dm1, sums, acc);
                else dt_collect<4, MT, BF16>(td, dm0, dm1, sums, acc);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) ds_mbar_arrive(ds_smem(&sh.taken[at.d().at]));
                const DsOp& op = P.ops[d.x & (DS_MAX_PHASE_OPS - 1)];
                ds_commit<MT>(acc, op.dst, (d.x & DS_DESC_FIRST) ? op.res : nullptr, op.res_plain != 0, (int)d.z * DT_ROWS + quarter * 32 + lane, op.N, M);
            }
            if constexpr (RO::TEAMS == 2) turn ^= 1u;
            else turn = turn + 1 == RO::TEAMS ? 0u : turn + 1;
            at.next();
        }
    }

    // -- buffers no phase reads (and the last outputs): float32 copies for the caller, one chunk per warp --
    if (*reinterpret_cast<volatile int*>(&sh.abort_flag) == 0) {
#pragma unroll 1
        for (int e = (int)blockIdx.x + (int)gridDim.x * cwarp; e < a.n_tails; e += (int)gridDim.x * RO::COLLECT_WARPS) {   // (few chunks: one per SM)
            const DsTail T = a.tails[e];                           // (n is a multiple of 4)
            DsQuad q[DS_TAIL_CHUNK / 128];
#pragma unroll
            for (int u = 0; u < DS_TAIL_CHUNK / 128; ++u)
                if (lane * 4 + 128 * u < T.n) ds_ld_quad(T.src + lane * 4 + 128 * u, q[u]);
#pragma unroll
            for (int u = 0; u < DS_TAIL_CHUNK / 128; ++u) {
                const int i = lane * 4 + 128 * u;
                if (i >= T.n || !ds_quad_complete(T.src + i, q[u], T.expect, wait_ns, &sh.abort_flag)) break;
                const float4 v = ds_quad_value(q[u]);
                *reinterpret_cast<float4*>(T.out + i) = v;
                if (a.out != nullptr) {
                    const int64_t o = (T.src - a.out_src) + i;
                    float unused;
                    if (o >= 0 && o < a.out_n) *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(a.out) + o) = ds_round4<BF16>(v, &unused);
                }
            }
        }
    }
    }   // (collect warps)

    // after a failed wait copies and tensor-core instructions may still be at work in this CTA: give them time
    if (*reinterpret_cast<volatile int*>(&sh.abort_flag)) __nanosleep(500000);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(512) : "memory");
    }
}

// ---- host: plan, cache, launch -----------------------------------------------------
namespace {

struct DecodePlan {
    std::vector<uint8_t> key;
    std::vector<aq_handle_t> handles;
    uint8_t* dev = nullptr;       // [phase records][ops][slab offsets][tail chunks][per-CTA phase tables][units per CTA]
    size_t feed_at = 0, xoff_at = 0, tails_at = 0, ctab_at = 0, total_at = 0;   // (the phase records are at 0)
    int n_ops = 0;
    int n_phases = 0;
    int n_tails = 0;
    bool late = false;            // ds_late, ds_teams of its phases
    int teams = 2;
    int device = 0;
    bool pinned = false;          // recorded into a CUDA graph: its device tables must outlive the plan cache's turnover
    std::vector<char> in_tails;   // per buffer: the tail chunks convert it (no phase reads it)
    uint64_t stamp = 0;
};

std::mutex g_plan_mutex;
std::vector<DecodePlan*> g_plans;
uint64_t g_plan_clock = 0;
constexpr size_t MAX_PLANS = 256;   // (a program with attention between its linears is one plan per stretch of linears)
u64 g_wait_ns = DS_WAIT_NS_DEFAULT;
bool g_hold = false;          // testing: the first packed input of a program expects one contribution too many

void drop_plan(DecodePlan* p) {
    if (p->dev) cudaFree(p->dev);
    delete p;
}

template <typename T> void key_put(std::vector<uint8_t>& k, const T& v) {
    const uint8_t* b = reinterpret_cast<const uint8_t*>(&v);
    k.insert(k.end(), b, b + sizeof(T));
}

}  // namespace

// How the units of the ops of one phase are dealt to the CTAs.  Every op's units are dealt on their own: with n = q G + r
// units and G CTAs, row s of the table takes q + 1 units if s < r, else q; an op starts `rot` rows further on than the first
// one, so that the odd units do not always land on the same CTAs.  It depends on the shapes alone, so the phases of equal
// blocks share a table (made anew for each of them it was most of a program's first call).
struct DealTable {
    struct Op { int NT8, KP, q, r, rot; };
    std::vector<Op> deal;
    std::vector<DsCtaPhase> cta;    // [row]
    std::vector<int16_t> xoff;      // [op][row]
    int turn = 0;                   // rows the next phase starts further on
    bool fits = false;              // no row needs more staged slabs than there is room for
};
// The table of ops[0 .. count), made if there is none yet; null when the kernel cannot take such a phase at all.
const DealTable* deal_table(std::vector<DealTable>& tables, const aq_stack_op_t* ops, int count, int n_cta) {
    DealTable t;
    int64_t all = 0;
    for (int i = 0; i < count; ++i) {
        const aq_handle_s* h = ops[i].w;
        const int NT8 = (h->NT + DS_FRAGS - 1) / DS_FRAGS;
        const int64_t nu = (int64_t)h->KP * NT8;
        all += nu;
        if (all > (int64_t)1 << 26 || h->KP > DS_MAX_CONTRIB) return nullptr;
        t.deal.push_back({NT8, h->KP, (int)(nu / n_cta), (int)(nu % n_cta), t.turn});
        t.turn = (int)((t.turn + nu % n_cta) % n_cta);
    }
    for (const DealTable& o : tables) {
        bool same = o.deal.size() == t.deal.size();
        for (size_t i = 0; i < t.deal.size() && same; ++i) same = o.deal[i].NT8 == t.deal[i].NT8 && o.deal[i].KP == t.deal[i].KP;
        if (same) return &o;
    }
    t.cta.resize(n_cta);
    t.xoff.assign((size_t)count * n_cta, 0);
    t.fits = true;
    for (int c = 0; c < n_cta && t.fits; ++c) {
        // the slabs the row reads, ascending, and where each op's first slab sits among them (an op's slabs are consecutive)
        DsCtaPhase& T = t.cta[c];
        memset(&T, 0, sizeof(T));
        std::vector<int> need;
        int lo[DS_MAX_PHASE_OPS];
        for (int i = 0; i < count && t.fits; ++i) {
            const DealTable::Op& d = t.deal[i];
            const int sl = (c + d.rot) % n_cta, u0 = d.q * sl + std::min(sl, d.r), u1 = u0 + d.q + (sl < d.r ? 1 : 0);
            T.total += u1 - u0;
            lo[i] = u0 / d.NT8;
            if (u0 == u1) continue;
            const int hi = (u1 - 1) / d.NT8;
            if (hi - lo[i] >= DS_MAX_SLOTS) t.fits = false;
            else for (int x = lo[i]; x <= hi; ++x) need.push_back(x);
        }
        std::sort(need.begin(), need.end());
        need.erase(std::unique(need.begin(), need.end()), need.end());
        if ((int)need.size() > DS_MAX_SLOTS) t.fits = false;
        if (!t.fits) break;
        T.n_slots = (int32_t)need.size();
        for (size_t x = 0; x < need.size(); ++x) T.slab_of_slot[x] = need[x];
        for (int i = 0; i < count; ++i)
            t.xoff[(size_t)i * n_cta + c] = (int16_t)(std::lower_bound(need.begin(), need.end(), lo[i]) - need.begin() - lo[i]);
    }
    tables.push_back(std::move(t));
    return &tables.back();
}

// Device tables of a program: one record per phase (at most DS_MAX_PHASE_OPS ops that
// read the same input vector) and the list of buffers nobody reads.  False when the program
// does not fit this kernel.
bool build_decode_tables(const aq_stack_t* p, const StackPlan& plan, int M, int n_cta, uint8_t* ws,
                         std::vector<DsPhase>& phases, std::vector<DsTail>& tails, std::vector<DsCtaPhase>& ctab,
                         std::vector<DsFeedOp>& feed_ops, std::vector<int16_t>& xoff, std::vector<char>& in_tails, int op_first, int op_end) {
    if (M < 1 || M > AQ_DECODE_MAX_M || p->n_ops > 32000 || plan.pk_off.empty()) return false;
    phases.clear();
    tails.clear();
    ctab.clear();
    feed_ops.clear();
    xoff.clear();
    std::vector<DealTable> tables;
    std::vector<int> writer(p->n_bufs, -1);         // op that writes the buffer
    std::vector<char> whole(p->n_bufs, 0);          // every CTA has seen the whole buffer complete (a normalised input)
    std::vector<char> recorded(p->n_bufs, 0);       // some phase writes the caller's float32 copy
    auto packed = [&](int b) { return reinterpret_cast<u64*>(ws + plan.pk_off[b]); };
    auto plain = [&](int b) { return reinterpret_cast<float*>(ws + plan.buf_off[b]); };
    auto expect_of = [&](int b) { return (uint32_t)p->ops[writer[b]].w->KP; };
    // a launch that runs ops [op_first, op_end) of the program: what earlier launches of the pass wrote is complete (as
    // packed sums and as the caller's float32 copy) before this one starts
    for (int i = 0; i < op_first; ++i) {
        writer[p->ops[i].dst] = i;
        whole[p->ops[i].dst] = 1;
        recorded[p->ops[i].dst] = 1;
    }
    int rot = 0;   // where the next op's odd units start
    bool hold = g_hold;
    const int n_ph = (int)plan.phase_first.size();
    for (int ph = 0; ph < n_ph; ++ph) {
        const int pfirst = plan.phase_first[ph];
        const int plast = (ph + 1 < n_ph) ? plan.phase_first[ph + 1] : p->n_ops;
        if (pfirst < op_first || pfirst >= op_end) continue;
        if (plast > op_end) return false;   // (a launch ends where a phase ends)
        for (int first = pfirst; first < plast;) {
            // as many of the phase's ops (at most DS_MAX_PHASE_OPS) as leave every CTA's staged slabs inside the
            // shared-memory buffer; the rest of them form a further phase with the same input
            const aq_stack_op_t& f = p->ops[first];
            const int64_t K = p->buf_width[f.src];
            if (K > (int64_t)1 << 24 || n_cta > 32767) return false;
            DsPhase P;
            int count = std::min(plast - first, DS_MAX_PHASE_OPS);
            const DealTable* tab = nullptr;
            for (; count >= 1; --count) {
                tab = deal_table(tables, p->ops + first, count, n_cta);
                if (tab == nullptr) return false;
                if (tab->fits) break;
            }
            if (count < 1) return false;
            const int last = first + count;
            // CTA c takes row (c + rot) mod (number of CTAs) of the table
            memset(&P, 0, sizeof(P));
            ctab.insert(ctab.end(), tab->cta.begin() + rot, tab->cta.end());
            ctab.insert(ctab.end(), tab->cta.begin(), tab->cta.begin() + rot);
            for (int i = 0; i < count; ++i) {
                const aq_handle_s* h = p->ops[first + i].w;
                DsFeedOp f2;
                memset(&f2, 0, sizeof(f2));
                f2.frags = h->frags; f2.NT = h->NT;
                f2.units_q = tab->deal[i].q;
                f2.units_r_rot = tab->deal[i].r | (((tab->deal[i].rot + rot) % n_cta) << 16);
                f2.word0 = (uint32_t)i | ((uint32_t)h->bits << DS_DESC_BITS_SHIFT) | ((uint32_t)phases.size() << DS_DESC_PHASE_SHIFT);
                feed_ops.push_back(f2);
                const int16_t* x = tab->xoff.data() + (size_t)i * n_cta;
                xoff.insert(xoff.end(), x + rot, x + n_cta);
                xoff.insert(xoff.end(), x, x + rot);
            }
            rot = (rot + tab->turn) % n_cta;
            auto source = [&](int b, const u64*& sp, const float*& sf, float*& rec, uint32_t& ex) {
                if (writer[b] < 0) { sp = nullptr; sf = plain(b); rec = nullptr; ex = 0; return; }   // the program input
                sp = packed(b); sf = nullptr; ex = expect_of(b);
                rec = recorded[b] ? nullptr : plain(b);
                recorded[b] = 1;
            };
            source(f.src, P.src, P.src_f, P.rec, P.expect);
            if (hold && P.src) { P.expect += 1; hold = false; }   // (a count no row reaches: every CTA's wait runs out)
            if (f.in_op == AQ_IN_SILU_MUL) source(f.src2, P.src2, P.src2_f, P.rec2, P.expect2);
            if (f.in_op == AQ_IN_RMSNORM) whole[f.src] = 1;
            P.stage = ws + plan.in_off[first];
            P.K = (int32_t)K; P.in_op = f.in_op; P.op_count = count;
            // several tokens: the row norms come from per-CTA partial sums exchanged through the workspace (whole
            // rows read by every CTA are 8 M K bytes per CTA from the same lines of L2)
            P.norm = nullptr;
            if (f.in_op == AQ_IN_RMSNORM && M >= 3 && (int64_t)M * K > DS_WHOLE_ROWS && !plan.nm_off.empty() && plan.nm_off[pfirst] != 0 && n_cta <= AQ_NORM_MAX_CTAS)
                P.norm = reinterpret_cast<u64*>(ws + plan.nm_off[pfirst]);
            for (int i = first; i < last; ++i) {
                const aq_stack_op_t& o = p->ops[i];
                DsOp& d = P.ops[i - first];
                d.dst = packed(o.dst);
                d.N = (int32_t)o.w->N;
                d.res = nullptr;
                if (o.out_op == AQ_OUT_ADD) {
                    // the residual is read without a wait: it must be complete for every CTA when the phase starts,
                    // i.e. the program input (plain float32) or an input that every CTA has already read as a whole
                    // (a normalised one)
                    if (writer[o.res] < 0) { d.res = plain(o.res); d.res_plain = 1; }
                    else if (whole[o.res]) d.res = packed(o.res);
                    else return false;
                }
            }
            for (int i = first; i < last; ++i) writer[p->ops[i].dst] = i;
            phases.push_back(P);
            first = last;
        }
    }
    // what no phase has copied out for the caller
    in_tails.assign(p->n_bufs, 0);
    for (int b = 1; b < p->n_bufs; ++b) {
        if (writer[b] < op_first || recorded[b]) continue;   // (written by this launch, read by none of its phases)
        const int64_t n = (int64_t)M * p->buf_width[b];
        if (n % 4) return false;
        in_tails[b] = 1;
        for (int64_t i = 0; i < n; i += DS_TAIL_CHUNK) {
            DsTail t;
            memset(&t, 0, sizeof(t));
            t.src = packed(b) + i; t.out = plain(b) + i;
            t.n = (int32_t)std::min<int64_t>(DS_TAIL_CHUNK, n - i);
            t.expect = expect_of(b);
            tails.push_back(t);
        }
    }
    return true;
}

// Collect teams for M tokens.  Reading a unit's sums and adding them sets the pace from five tokens on, and a third team helps there;
// so do its threads where every CTA reads whole rows for the row norms and they save it a step (256 or 384 threads, a group of
// four elements each).  With three and four tokens it gains nothing where units set the pace and costs where boundaries do, and
// with seven and eight the same holds for whole rows of which it saves no step.  Measured, us with two / three teams: 18 expert
// blocks (K = 1024) 340 / 373 at 4 tokens, 402 / 396 at 5, 443 / 471 at 7, 457 / 482 at 8; 8 blocks of the 2B shape (2048) 270 / 289
// at 4, 355 / 341 at 5, 359 / 350 at 6, 386 / 395 at 7, 400 / 405 at 8; of the 7B shape (shares from 5 tokens on) 421 / 423 at 4,
// 525 / 492 at 5, 578 / 547 at 8; 8 blocks of 1280 / 5120 (two steps / one) 208 / 188 at 5, 242 / 224 at 8.
static int ds_teams(const std::vector<DsPhase>& phases, int M) {
    if (M <= 4) return 2;
    if (M <= 6) return 3;
    bool whole_rows = false;
    for (const DsPhase& P : phases) {
        if (P.in_op != AQ_IN_RMSNORM || P.norm != nullptr) continue;
        const int q4 = P.K / 4, two = DsRoles<2>::CTHREADS, three = DsRoles<3>::CTHREADS;
        if ((q4 + two - 1) / two != (q4 + three - 1) / three) return 3;
        whole_rows = true;
    }
    return whole_rows ? 2 : 3;
}
// Whether the operand of unit n + 2 is unpacked only when the sums of unit n have been read, not as soon as its instructions have
// completed.  At once is better where a phase is many units long; where it is not, unit n + 2 belongs to the next phase, and
// unpacking it takes issue slots from the sums that everybody is waiting for.  The line lies at the units a CTA meets of a phase, on
// average; us at once / late: two teams, 18 expert blocks (0.9 units) 285 / 272 at 2 tokens, 335 / 320 at 4, 474 / 457 at 8; 8 blocks
// of 2048 / 8192 (3.1) 212 / 209 at 4, 2304 / 8192 (3.5) 240 / 236, 2560 / 8192 (4.0) 245 / 243, 3072 / 8192 (5.0) 221 / 223 at 2, of
// the 7B shape (10) 344 / 348 at 2; three teams, 5 tokens: expert 407 / 396, 1536 / 6144 (1.7) 200.7 / 198.6, 2048 / 6144 (2.4) 248 /
// 251, 3072 / 8192 315 / 325, 7B shape 492 / 509.
static bool ds_late(int64_t units, int64_t cta_phases, int teams) { return units < (teams == 2 ? 4 : 2) * cta_phases; }

// What a pass needs before its first launch: x as float32 (groups of eight) and zeros in the packed sums.  One kernel in place of
// a conversion and a memset: a pass of a small program takes 15 us, and each launch before the big one added 1.5.
template <bool BF16>
__global__ void __launch_bounds__(256) begin_pass_kernel(const uint4* __restrict__ x, float4* __restrict__ out, int64_t n8, int rest, uint4* __restrict__ zero, int64_t zero16) {
    pdl_wait();
    const int64_t i0 = (int64_t)blockIdx.x * 256 + threadIdx.x, step = (int64_t)gridDim.x * 256;
    for (int64_t i = i0; i < n8; i += step) {
        const uint4 v = x[i];
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        float f[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float2 p;
            if constexpr (BF16) p = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[j]));
            else p = __half22float2(*reinterpret_cast<const __half2*>(&w[j]));
            f[2 * j] = p.x; f[2 * j + 1] = p.y;
        }
        out[2 * i] = make_float4(f[0], f[1], f[2], f[3]);
        out[2 * i + 1] = make_float4(f[4], f[5], f[6], f[7]);
    }
    if (i0 < rest) {   // elements past the last whole group
        const uint16_t u = reinterpret_cast<const uint16_t*>(x + n8)[i0];
        float f;
        if constexpr (BF16) f = __bfloat162float(__ushort_as_bfloat16(u));
        else f = __half2float(__ushort_as_half(u));
        reinterpret_cast<float*>(out + 2 * n8)[i0] = f;
    }
    for (int64_t i = i0; i < zero16; i += step) zero[i] = make_uint4(0, 0, 0, 0);
}

template <int MT, int TEAMS, bool BF16>
static cudaError_t launch_ds(const DsArgs& a, int grid, cudaStream_t s) {
    auto kern = decode_stack_kernel<MT, TEAMS, BF16>;
    static PerDeviceOnce configured;
    {
        const int rc = configured.run(current_device(), [&] {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DsShared));
            if (e != cudaSuccess) return (int)e;
            int per_sm = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, DsRoles<TEAMS>::THREADS, sizeof(DsShared));
            if (e != cudaSuccess) return (int)e;
            return per_sm < 1 ? (int)cudaErrorCooperativeLaunchTooLarge : 0;
        });
        if (rc != 0) return rc < 0 ? cudaErrorInvalidDevice : (cudaError_t)rc;
    }
    DsArgs args = a;
    void* params[1] = {&args};
    cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<void*>(kern), dim3((unsigned)grid), dim3(DsRoles<TEAMS>::THREADS), params,
                                                sizeof(DsShared), s);
    if (e == cudaSuccess) count_launch();
    return e;
}

// The part of a plan's key that depends on the program alone (ops, their matrices, buffer widths).
void decode_program_key(const aq_stack_t* p, std::vector<uint8_t>& key) {
    key.reserve(key.size() + (size_t)p->n_ops * (sizeof(aq_stack_op_t) + 8) + (size_t)p->n_bufs * 8 + 16);
    key_put(key, p->n_ops); key_put(key, p->n_bufs);
    for (int i = 0; i < p->n_ops; ++i) {
        key_put(key, p->ops[i]);
        key_put(key, p->ops[i].w->frags);
    }
    for (int b = 0; b < p->n_bufs; ++b) key_put(key, p->buf_width[b]);
}

int launch_decode_stack(const aq_stack_t* p, const StackPlan& plan, int M, aq_dtype_t dt, uint8_t* ws, cudaStream_t s,
                        cudaError_t* err, const void* x0, void* out, int out_buf, bool* wrote_out, int op_first, int op_end,
                        const std::vector<uint8_t>* program_key) {
    *err = cudaSuccess;
    *wrote_out = false;
    if (op_end < 0) op_end = p->n_ops;
    const int grid = sm_count();
    const int dev = current_device();
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) { cudaGetLastError(); cap = cudaStreamCaptureStatusNone; }
    const bool capturing = (cap != cudaStreamCaptureStatusNone);
    // key: everything the device tables are computed from
    std::vector<uint8_t> key;
    key_put(key, M); key_put(key, dev); key_put(key, grid); key_put(key, ws); key_put(key, op_first); key_put(key, op_end);
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    key_put(key, g_hold);
    if (program_key) key.insert(key.end(), program_key->begin(), program_key->end());   // (built once for all the launches of a pass)
    else decode_program_key(p, key);

    DecodePlan* dp = nullptr;
    for (DecodePlan* q : g_plans)
        if (q->key == key) { dp = q; break; }
    if (!dp) {
        if (capturing) return 1;   // tables are built (allocation, synchronous copies) by an eager call only
        std::vector<DsPhase> phases;
        std::vector<DsTail> tails;
        std::vector<DsCtaPhase> ctab;
        std::vector<DsFeedOp> feed_ops;
        std::vector<int16_t> xoff;
        std::vector<char> in_tails;
        if (!build_decode_tables(p, plan, M, grid, ws, phases, tails, ctab, feed_ops, xoff, in_tails, op_first, op_end)) return 1;
        if (g_plans.size() >= MAX_PLANS) {   // make room: the oldest plan no graph refers to
            size_t oldest = g_plans.size();
            for (size_t i = 0; i < g_plans.size(); ++i)
                if (!g_plans[i]->pinned && (oldest == g_plans.size() || g_plans[i]->stamp < g_plans[oldest]->stamp)) oldest = i;
            if (oldest == g_plans.size()) return 1;   // all pinned: this program runs op by op
            drop_plan(g_plans[oldest]);
            g_plans.erase(g_plans.begin() + oldest);
        }
        dp = new DecodePlan();
        dp->key = key;
        dp->device = dev;
        for (int i = 0; i < p->n_ops; ++i) dp->handles.push_back(p->ops[i].w);
        dp->in_tails = in_tails;
        dp->n_phases = (int)phases.size();
        dp->n_tails = (int)tails.size();
        // one table after the other, each at a multiple of 256 bytes
        std::vector<uint8_t> image;
        image.reserve(phases.size() * sizeof(DsPhase) + (feed_ops.size() + 1) * (sizeof(DsFeedOp) + 2 * grid) + tails.size() * sizeof(DsTail) + ctab.size() * sizeof(DsCtaPhase) + 4096);
        auto add = [&](const void* data, size_t bytes) {
            const size_t at = image.size();
            image.resize((at + bytes + 255) / 256 * 256);
            if (bytes) memcpy(image.data() + at, data, bytes);
            return at;
        };
        std::vector<int32_t> unit_total(grid, 0);
        for (size_t i = 0; i < ctab.size(); ++i) unit_total[i % grid] += ctab[i].total;
        dp->teams = ds_teams(phases, M);
        dp->late = ds_late(std::accumulate(unit_total.begin(), unit_total.end(), (int64_t)0), (int64_t)phases.size() * grid, dp->teams);
        dp->n_ops = (int)feed_ops.size();
        feed_ops.push_back(DsFeedOp{});   // (the feeder reads one op ahead)
        xoff.resize(xoff.size() + grid, 0);
        add(phases.data(), phases.size() * sizeof(DsPhase));
        dp->feed_at = add(feed_ops.data(), feed_ops.size() * sizeof(DsFeedOp));
        dp->xoff_at = add(xoff.data(), xoff.size() * sizeof(int16_t));
        dp->tails_at = add(tails.data(), tails.size() * sizeof(DsTail));
        dp->ctab_at = add(ctab.data(), ctab.size() * sizeof(DsCtaPhase));
        dp->total_at = add(unit_total.data(), unit_total.size() * sizeof(int32_t));
        cudaError_t e = cudaMalloc(&dp->dev, image.size());
        if (e == cudaSuccess) e = cudaMemcpy(dp->dev, image.data(), image.size(), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) { cudaGetLastError(); drop_plan(dp); *err = e; return -1; }
        g_plans.push_back(dp);
    }
    dp->stamp = ++g_plan_clock;
    if (capturing) dp->pinned = true;

    DsArgs a;
    a.phases = reinterpret_cast<const DsPhase*>(dp->dev);
    a.feed_ops = reinterpret_cast<const DsFeedOp*>(dp->dev + dp->feed_at);
    a.xoff = reinterpret_cast<const int16_t*>(dp->dev + dp->xoff_at);
    a.unit_total = reinterpret_cast<const int32_t*>(dp->dev + dp->total_at);
    a.n_ops = dp->n_ops;
    a.tails = reinterpret_cast<const DsTail*>(dp->dev + dp->tails_at);
    a.ctab = reinterpret_cast<const DsCtaPhase*>(dp->dev + dp->ctab_at);
    a.n_phases = dp->n_phases;
    a.n_tails = dp->n_tails;
    a.M = M;
    a.late = dp->late ? 1 : 0;
    a.wait_ns = g_wait_ns;
    a.out = nullptr; a.out_src = nullptr; a.out_n = 0;
    if (out != nullptr && out_buf >= 1 && out_buf < p->n_bufs && dp->in_tails[out_buf] &&
        (reinterpret_cast<uintptr_t>(out) & 7u) == 0) {
        a.out = out;
        a.out_src = reinterpret_cast<const u64*>(ws + plan.pk_off[out_buf]);
        a.out_n = (int64_t)M * p->buf_width[out_buf];
        *wrote_out = true;
    }
    // once per pass: the input widened, and the packed sums zeroed (a later launch reads what the earlier ones left)
    cudaError_t e = cudaSuccess;
    if (x0) {
        const int64_t n0 = (int64_t)M * p->buf_width[0], n8 = n0 / 8, zero16 = (int64_t)(plan.pk_end - plan.pk_begin) / 16;
        const unsigned blocks = (unsigned)std::min<int64_t>((std::max(n8, zero16) + 511) / 512, 4 * grid);
        float4* widened = reinterpret_cast<float4*>(ws + plan.buf_off[0]);
        uint4* zero = reinterpret_cast<uint4*>(ws + plan.pk_begin);
        if (dt == AQ_BF16) e = launch_pdl(begin_pass_kernel<true>, dim3(blocks), dim3(256), 0, s, (const uint4*)x0, widened, n8, (int)(n0 - 8 * n8), zero, zero16);
        else e = launch_pdl(begin_pass_kernel<false>, dim3(blocks), dim3(256), 0, s, (const uint4*)x0, widened, n8, (int)(n0 - 8 * n8), zero, zero16);
        count_launch();
    }
    if (e == cudaSuccess) {
        const bool bf = (dt == AQ_BF16);
        if (M == 1) e = bf ? launch_ds<1, 2, true>(a, grid, s) : launch_ds<1, 2, false>(a, grid, s);
        else if (M == 2) e = bf ? launch_ds<2, 2, true>(a, grid, s) : launch_ds<2, 2, false>(a, grid, s);
        else if (M <= 4) e = bf ? launch_ds<4, 2, true>(a, grid, s) : launch_ds<4, 2, false>(a, grid, s);
        else if (dp->teams == 2) e = bf ? launch_ds<8, 2, true>(a, grid, s) : launch_ds<8, 2, false>(a, grid, s);
        else e = bf ? launch_ds<8, 3, true>(a, grid, s) : launch_ds<8, 3, false>(a, grid, s);
    }
    if (e != cudaSuccess) { *err = e; return -1; }
    return 0;
}

void decode_stack_forget(aq_handle_t h) {
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    for (size_t i = 0; i < g_plans.size();) {
        bool uses = false;
        for (aq_handle_t x : g_plans[i]->handles)
            if (x == h) { uses = true; break; }
        if (uses) { drop_plan(g_plans[i]); g_plans.erase(g_plans.begin() + i); }
        else ++i;
    }
}

int read_decode_status(bool clear) {
    int v = 0;
    cudaMemcpyFromSymbol(&v, g_decode_status, sizeof(int));
    if (clear && v) { int z = 0; cudaMemcpyToSymbol(g_decode_status, &z, sizeof(int)); }
    return v;
}

void set_decode_hold(bool on) {
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    g_hold = on;
}

void set_decode_wait_ns(unsigned long long ns) {
    std::lock_guard<std::mutex> lock(g_plan_mutex);
    g_wait_ns = ns ? ns : DS_WAIT_NS_DEFAULT;
}

}  // namespace aq
