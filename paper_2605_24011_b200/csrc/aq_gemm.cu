// Prefill path (M > 8): dequantise-to-half + tensor-core GEMM on the packed
// weights, out[m][n] = (res[m][n]) + sum_k x[m][k] w_hat[n][k]  (Appendix D:
// dequantise on the fly inside the low-bit kernel; Eq. 1 for the decode).
//
// Both operands enter the tensor core as binary16: a dequantised weight is
// fp16(scale * q + min) (one half-precision FMA, 11 significant bits, so the
// worst case of the product sum is 2^-11 sum|x w|).  bfloat16 activations are
// widened to binary16 by the caller of this kernel (exact wherever the value is
// inside binary16's range; a token row that is not comes scaled by a power of
// two, undone in the epilogue through tok_scale).
//
// Bound: by its flops the tensor cores (dense contraction, 2 M flops per weight).  In
// fact no unit is full: 11008 x 4096 at 512 tokens (pairs, 86 tiles on 74 of them) keeps
// the tensor pipe 51 % active, L2 at 21 % of its rate, issue slots at 26 % (single CTAs: 47,
// 20 and 38 %); the start (4 us to the first instruction), drains of 128 KB per SM and
// pieces of tiles added through L2 share the rest.  With few tokens it is the chain of
// latencies from launch to sums (2.7 us), epilogue and adds.
//
// tcgen05 UMMA, 256 weight rows x up to 128 tokens per tile:
//   A (M side, 2 x 128) = weight rows, dequantised by sixteen warps from the packed
//                       fragments straight into TMEM (tcgen05.st): two row halves
//                       of 64 k are a stage of 64 columns, four stages,
//   B (N side, <=128) = tokens, fetched by TMA (128-byte swizzle); one token tile
//                       serves both row halves,
//   D[2][128 lanes][tokens] fp32 in TMEM; with up to 64 tokens two sets of them.
// Why this shape.  With the dequantised tile in shared memory and 128 x 512 tiles
// the loop was bound by moving operands (per 128 x 256 x 128 of work 96 KB read by
// the tensor core, 64 KB of tokens and 16 KB of weights written: 0.875 us against
// 0.54 us of tensor time).  Here the same work writes 32 KB of tokens and reads 64,
// and half the token bytes come out of L2; the price is that a weight is dequantised
// once per 128 tokens instead of once per 512.  Measured, that design / this one: 18 blocks
// of a 2B model at 768 tokens 4.96 / 4.51 ms, 32 of a 7B model at 512 tokens 8.75 / 8.28 ms,
// 18 of a 300M expert at 50 tokens 931 / 678 us, one 11008 x 4096 matrix at 200 tokens
// 49.2 / 30.8 us (with the zeroing rule at gemm_stores_first and the cast by finalize_kernel).
//
// Large products run on CTA pairs (tcgen05 cta_group::2, one instruction over 256 rows and up to 256 tokens; each CTA
// dequantises its 128 rows and holds half of the tokens): half the dequantisation, half the packed bytes and half the
// operand reads from shared memory per flop.  In an instrumented copy 64 k of a tile (512 cycles of instructions) take 595
// cycles instead of 880; products gain 5 to 12 %, a 7B-shaped pass of 512 tokens 3 to 4 %.  22016 x 4096 at 512 tokens: 1190
// TFLOP/s over 50 ms, 1029 over 5 s, when the chip is at its power limit (985 W, 1.61 GHz of 1.97; cuBLAS 1593 and 1359, 1.31
// GHz).  Deeper rings (4 to 7 token slots, 4 to 7 epilogue chunks per warp) change nothing.
//
// One persistent CTA, or pair, per SM (or two).  The work -- (row tile, token tile, 128-k slab)
// triples -- is cut into contiguous runs, one per CTA, balanced for slabs plus a
// fixed cost per piece of a tile; a run that covers a tile's whole K stores its
// sums, any other run adds them (reduce-add copies; see the store-first protocol
// below).
// Warp roles: 0..15 = dequantise, 16..19 = epilogue, 20 = token-tile TMA producer
// (+ TMEM allocation), 21 = MMA issue, 22 = packed-fragment bulk-copy producer.
// Epilogue: TMEM -> registers -> 32 x 32 fp32 chunks in shared memory -> TMA tensor
// store, or TMA reduce-add when the tile is split; the next tile's instructions
// start when TMEM has been read, not when the copies have drained.  Every mbarrier
// wait is bounded; when one runs out the CTA raises a status word, drains and returns.
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <vector>

#include "aq_gemm_runs.h"
#include "aq_internal.h"
#include "aq_layout.cuh"
#include "aq_tc.cuh"
#include "aq_tmem.cuh"

namespace aq {

constexpr int GM_ROWS = 256;       // weight rows per tile: two instructions of one CTA, or one instruction of a CTA pair
constexpr int GM_FRAGS = GM_ROWS / ROWS;
constexpr int GM_KSTAGE = 64;      // k per stage (one 128-byte swizzle atom of 16-bit elements)
constexpr int GM_ACOL0 = 256;      // first TMEM column of the dequantised stages; D lies below
constexpr int GM_PSTAGES = 4;      // packed-fragment ring (one k-slab of 128 per slot)
constexpr int GM_DQ_WARPS = 16, GM_EP_WARPS = 4;
constexpr int GM_EP0 = GM_DQ_WARPS, GM_TMA = GM_EP0 + GM_EP_WARPS, GM_MMA = GM_TMA + 1, GM_PACKED = GM_MMA + 1;
constexpr int GM_WARPS = 24;       // (one idle: registers are dealt to groups of four)
constexpr int GM_THREADS = GM_WARPS * 32;
// Registers per thread by role, out of the 80 the block is launched with
constexpr int GM_REGS = 80, GM_REGS_DQ = 72, GM_REGS_EP = 128, GM_REGS_OTHER = 64;
static_assert(GM_DQ_WARPS * GM_REGS_DQ + GM_EP_WARPS * GM_REGS_EP + 4 * GM_REGS_OTHER <= GM_WARPS * GM_REGS && GM_THREADS * GM_REGS <= 65536, "the roles' registers fit");

// What depends on whether a tile belongs to one CTA or to a pair of them.
template <bool PAIR> struct Tile {
    static constexpr int FRAGS = PAIR ? GM_FRAGS / 2 : GM_FRAGS;   // 16-row tiles a CTA dequantises
    static constexpr int MAX_TN = PAIR ? GM_PAIR_TOKENS : GM_TOKENS;   // tokens per tile (UMMA N)
    static constexpr int B_BYTES = 128 * 128;                      // token slot: 128 tokens x 64 k (of a pair each CTA holds half of the tile's tokens)
    static constexpr int B_SLOTS = PAIR ? 7 : 5;
    static constexpr int P_BYTES = FRAGS * frag_bytes(4);          // packed fragments of one slab (largest width)
    // Dequantise warps: groups take the k-slabs in turn, two fragments per warp (with one group of sixteen a slab took as long
    // as one warp's chain of waits).  Both rings have whole numbers of slots per group, so a group meets every use of the
    // slots it works on (a barrier only tells a phase from the one before it).
    static constexpr int DQ_GROUP = FRAGS / 2, DQ_GROUPS = GM_DQ_WARPS / DQ_GROUP;
    static constexpr int A_STAGES = 2 * DQ_GROUPS;                 // dequantised stages in TMEM
    static constexpr int A_COLS = FRAGS * 4;                       // TMEM columns of one: [row half][32]
    static constexpr int CHUNKS = 4;                    // epilogue chunks per warp
    static constexpr int STG_BYTES = GM_EP_WARPS * CHUNKS * 4096;
    static constexpr int SMEM = 1024 + B_SLOTS * B_BYTES + GM_PSTAGES * P_BYTES + STG_BYTES + 512;
    static_assert(GM_PSTAGES % DQ_GROUPS == 0 && GM_ACOL0 + A_STAGES * A_COLS <= 512 && SMEM <= 227 * 1024, "slots belong to groups; fits an SM");
};
constexpr uint32_t GM_SPIN_LIMIT = 40u * 1000u * 1000u;

__device__ int g_gemm_status = 0;  // nonzero: a bounded wait ran out (code = which)

// Split tiles without zeroing the output first: the run that holds a tile's last k-slab is the first thing its CTA
// does; it STORES its sums and then writes the launch's epoch into the tile's flags; the other runs of the tile add
// theirs once they see it.  One flag per epilogue warp: a warp adds to the rows that the warp of the same TMEM quarter
// stored, so no warp of a CTA waits for another (a barrier between them would not end when one of them has given up).
// Flags are never reset: every launch has its own epoch and takes the next of a few arrays.
constexpr int GM_FLAG_SLOTS = 8;
constexpr int GM_MAX_TILES = 8192;
__device__ uint32_t g_tile_flags[GM_FLAG_SLOTS][GM_MAX_TILES][2 * GM_EP_WARPS];   // (the second half: the odd CTA of a pair)
static std::atomic<bool> g_gemm_hold{false};   // testing: launches leave their flags down

constexpr int GM_MAX_OPS = 4;      // matrices that share one input (q|k|v, gate|up) run as one launch

struct GemmOp {
    const uint8_t* frags;
    float* out;            // float32 [M][ldo]
    const float* res;      // float32 [M][ldo] added once, or null
    int64_t ldo;
    int N;
    int NT;                // 16-row tiles
    int R;                 // row tiles of 256
    int bits;
};

struct GemmArgs {
    GemmOp op[GM_MAX_OPS];
    int n_ops;
    int M;
    int n_slabs;           // 128-k slabs (K padded to 256)
    int n_st;              // token tiles
    int tn;                // tokens per tile (the last may hold fewer)
    int tma_out;           // 1: the epilogue writes through the output tensor maps (needs ldo % 4 == 0)
    int store_first;       // 1: split tiles of matrices without a residual use the store-then-add protocol above
    int flag_slot;
    uint32_t epoch;
    int hold;              // testing: flags stay down
    const float* tok_scale;    // per token: the power of two its row of x was divided by, or null
    int bounds[GM_MAX_GRID + 1];   // CTA (or pair) c works on half slabs [bounds[c], bounds[c + 1]) (even numbers)
};

struct GemmOutMaps { CUtensorMap m[GM_MAX_OPS]; };

// One contiguous piece of a CTA's run: slabs [s0, s1) of tile (rt, st).
struct GemmSeg {
    int op, rt, st, s0, s1;   // rt: row tile inside matrix op
    int tile;                 // index of the tile in the launch
    int w;                    // its tokens, rounded up to 16 (a pair: 32)
    int n_rt;                 // the CTA's 16-row tiles (1..16; of a pair 0..8)
};

// Tiles are ordered by matrix, row tile, token tile: a CTA that goes on to the next token tile finds the packed rows in L2.
template <bool PAIR>
__device__ __forceinline__ bool gemm_next_seg(int& pos, int hi, const GemmArgs& a, int rank, GemmSeg& sg) {
    if (pos >= hi) return false;
    const int c1 = 2 * a.n_slabs;
    const int t = pos / c1, end = min(hi, (t + 1) * c1);
    sg.s0 = (pos - t * c1) >> 1; sg.s1 = (end - t * c1) >> 1;
    pos = end;
    sg.tile = t;
    int r = t / a.n_st;
    sg.st = t - r * a.n_st;
    sg.op = 0;
    while (sg.op + 1 < a.n_ops && r >= a.op[sg.op].R) { r -= a.op[sg.op].R; ++sg.op; }
    sg.rt = r;
    sg.w = min(a.tn, (a.M - sg.st * a.tn + (PAIR ? 31 : 15)) & ~(PAIR ? 31 : 15));
    sg.n_rt = min(Tile<PAIR>::FRAGS, a.op[sg.op].NT - r * GM_FRAGS - rank * Tile<PAIR>::FRAGS);
    if (PAIR) sg.n_rt = max(0, sg.n_rt);
    return true;
}

template <bool PAIR>
__device__ __forceinline__ void give_up(volatile int* abort_flag, int code) {
    *abort_flag = 1;
    if constexpr (PAIR) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_map(smem_u32((const void*)abort_flag), cluster_rank() ^ 1u)), "r"(1) : "memory");
    atomicCAS(&g_gemm_status, 0, code);
}
// Bounded wait.  Returns false when the limit ran out or another role (of either CTA of a pair) gave up.  OWN: every arrival comes from
// this CTA; of a pair the others may come from its partner, so they are waited for at cluster scope (0 to 1 % of a product).
template <bool PAIR, bool OWN = !PAIR>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int code) {
    for (uint32_t i = 0; i < GM_SPIN_LIMIT; ++i) {
        if (OWN ? mbar_try(bar, parity) : mbar_try_cluster(bar, parity)) return true;
        if (i > 2000) {
            __nanosleep(40);
            if (*abort_flag) return false;
        }
    }
    give_up<PAIR>(abort_flag, code);
    return false;
}
template <bool PAIR, bool OWN = !PAIR>
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int code) {
    return __all_sync(0xffffffffu, mbar_wait<PAIR, OWN>(bar, parity, abort_flag, code));
}
// Arrive on a barrier of the CTA that issues the instructions: given as a cluster address for a pair, as a local one otherwise.
template <bool PAIR>
__device__ __forceinline__ void arrive_issuer(uint32_t bar) {
    if constexpr (PAIR) mbar_arrive_cluster(bar);
    else mbar_arrive(bar);
}
// Barriers of the CTA, or of both CTAs of the pair, count the instructions issued so far.
template <bool PAIR>
__device__ __forceinline__ void commit_all(uint32_t bar) {
    if constexpr (PAIR) umma_commit_both(bar);
    else umma_commit(bar);
}

// Pair (codes 2i, 2i + 1) of block j, row half hi as two dequantised weights.  The codes are OR-ed, where they lie, into the
// mantissa of the binary16 constant whose last place is worth 2^-pos (1024 at position 0, 64 at 4, ...); subtracting it is
// exact and leaves the codes; one half2 FMA with scale and min.
template <int BITS>
__device__ __forceinline__ uint32_t dequant_pair(const InPlace<BITS>& ip, int f, int r, uint32_t dm) {
    const uint32_t magic = 0x64006400u - (uint32_t)(InPlace<BITS>::pos(f)) * 0x04000400u;   // 2^(10 - pos)
    const uint32_t p = ip.reg_or(f, r, magic);
    const __half2 q = __hsub2(*reinterpret_cast<const __half2*>(&p), *reinterpret_cast<const __half2*>(&magic));
    const __half2 v = *reinterpret_cast<const __half2*>(&dm);
    const __half2 w = __hfma2(q, __low2half2(v), __high2half2(v));
    return *reinterpret_cast<const uint32_t*>(&w);
}

// One dequantise warp's share of a k-slab: two neighbouring fragments (32 rows x 128 k) as lanes of two A stages.  n_have of
// them exist (past the end of the matrix nothing is written: those rows of D are not stored).  Returns false when a wait
// ran out.
template <int BITS, bool PAIR>
__device__ __forceinline__ bool dequant_slab(const uint8_t* frags, int n_have, int lane, uint32_t tmem_a, uint32_t bar_pempty_slot,
                                             uint32_t bar_aempty, uint32_t bar_afull, uint32_t parity, volatile int* abort_flag) {
    const int g = lane >> 2;
    // (absent fragments: whatever the slot holds)
    LaneCodes<BITS> lc[2];
    uint4 s0[2], s1[2];   // half2 (scale, min) of rows g, g + 8
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint8_t* f = frags + i * frag_bytes(BITS);
        load_lane_codes<BITS>(lc[i], f, lane);
        s0[i] = *reinterpret_cast<const uint4*>(f + g * 16);
        s1[i] = *reinterpret_cast<const uint4*>(f + (g + 8) * 16);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!mbar_wait_warp<PAIR>(bar_aempty + 8 * h, parity ^ 1, abort_flag, 6)) return false;
        tc_fence_after();
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            InPlace<BITS> ip;
            ip.prepare(lc[i]);
            const uint32_t dm[2][4] = {{s0[i].x, s0[i].y, s0[i].z, s0[i].w}, {s1[i].x, s1[i].y, s1[i].z, s1[i].w}};
            uint32_t v[16];
#pragma unroll
            for (int f = 0; f < 4; ++f)
#pragma unroll
                for (int r = 0; r < 4; ++r) v[4 * f + r] = dequant_pair<BITS>(ip, 4 * h + f, r, dm[r & 1][2 * h + (f >> 1)]);
            if (i < n_have) tmem_st_16x128(tmem_a + h * Tile<PAIR>::A_COLS + ((uint32_t)(i * 16) << 16), v);
            else if (h == 1 && i == 0) asm volatile("" ::"r"(v[0]));
        }
        if (h == 1) {
            // The packed slot is given back only here: its refill is written through the asynchronous proxy, which may
            // overtake shared-memory loads that have been issued but not returned.  By now every lane has used what it
            // loaded (lanes of absent fragments read nothing that matters).
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_pempty_slot);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_issuer<PAIR>(bar_afull + 8 * h);
    }
    return true;
}

template <bool PAIR>
__global__ void __launch_bounds__(GM_THREADS, 1) gemm_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ GemmOutMaps tmap_out, const __grid_constant__ GemmArgs a) {
    using T = Tile<PAIR>;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* sB = smem;
    uint8_t* sP = sB + T::B_SLOTS * T::B_BYTES;
    uint8_t* sC = sP + GM_PSTAGES * T::P_BYTES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sC + T::STG_BYTES);
    const uint32_t bar_afull = smem_u32(bars), bar_aempty = bar_afull + 8 * T::A_STAGES;
    const uint32_t bar_bfull = bar_aempty + 8 * T::A_STAGES, bar_bempty = bar_bfull + 8 * T::B_SLOTS;
    const uint32_t bar_pfull = bar_bempty + 8 * T::B_SLOTS, bar_pempty = bar_pfull + 8 * GM_PSTAGES;
    const uint32_t bar_dfull = bar_pempty + 8 * GM_PSTAGES, bar_dempty = bar_dfull + 16;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * T::A_STAGES + 2 * T::B_SLOTS + 2 * GM_PSTAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    // Of a pair both CTAs take rows (rank 0 the first 128 of the tile) and half of the tokens; rank 0 issues the instructions,
    // and its afull, bfull and dempty collect both CTAs' arrivals.
    const int rank = PAIR ? (int)cluster_rank() : 0, run = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;
    // sets of accumulators (128 columns each, where two fit), columns of a row half
    const int n_buf = a.tn <= T::MAX_TN / 2 ? 2 : 1, d_cols = a.tn <= 64 ? 64 : 128;

    if (threadIdx.x == 0) {
        constexpr int N = PAIR ? 2 : 1;
        for (int s = 0; s < T::A_STAGES; ++s) { mbar_init(bar_afull + 8 * s, N * T::DQ_GROUP); mbar_init(bar_aempty + 8 * s, 1); }
        for (int s = 0; s < T::B_SLOTS; ++s) { mbar_init(bar_bfull + 8 * s, 1); mbar_init(bar_bempty + 8 * s, 1); }
        for (int s = 0; s < GM_PSTAGES; ++s) { mbar_init(bar_pfull + 8 * s, 1); mbar_init(bar_pempty + 8 * s, T::DQ_GROUP); }
        for (int s = 0; s < 2; ++s) { mbar_init(bar_dfull + 8 * s, 1); mbar_init(bar_dempty + 8 * s, N * GM_EP_WARPS); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == GM_TMA) {
        if constexpr (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(512) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "n"(512) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (PAIR) cluster_sync_all();   // the partner's barriers exist before anything is counted on them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // The packed weights never change, so their copies and the dequantisation start at once, under the tail of the
    // kernel before this one; the roles that read or write activations (token tiles, epilogue) call pdl_wait() first.
    pdl_launch_dependents();

    GemmSeg sg;
    int pos = a.bounds[run];
    const int run_hi = a.bounds[run + 1];

    if (warp < GM_DQ_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(GM_REGS_DQ));
        // ---------------- dequantise ------------------------------------------------------------------
        // TMEM lanes 32 quarter .. + 31 of row half rh: fragments 8 rh + 2 quarter and the next of the tile
        const int quarter = warp & 3, rh = PAIR ? 0 : (warp >> 2) & 1, group = warp / T::DQ_GROUP, ft = 8 * rh + 2 * quarter;
        const uint32_t tmem_a = tmem_base + GM_ACOL0 + (uint32_t)(group * 2 * T::A_COLS + rh * 32) + ((uint32_t)(quarter * 32) << 16);
        const uint32_t af_pair = PAIR ? cluster_map(bar_afull + 16 * group, 0) : 0;
        uint32_t n = 0;   // slabs of the run so far
        bool ok = true;
        while (ok && gemm_next_seg<PAIR>(pos, run_hi, a, rank, sg)) {
            const int bits = a.op[sg.op].bits;
            const int n_have = min(2, sg.n_rt - ft);
            for (int s = sg.s0; s < sg.s1 && ok; ++s, ++n) {
                if ((int)(n % T::DQ_GROUPS) != group) continue;
                const uint32_t ps = n % GM_PSTAGES, parity = (n / T::DQ_GROUPS) & 1;   // (of the group's two A stages)
                ok = mbar_wait_warp<PAIR, true>(bar_pfull + 8 * ps, (n / GM_PSTAGES) & 1, abort_flag, 5);
                if (!ok) break;
                const uint8_t* frags = sP + ps * T::P_BYTES + ft * frag_bytes(bits);
                const uint32_t ae = bar_aempty + 16 * group, af = PAIR ? af_pair : bar_afull + 16 * group;
                if (bits == 2) ok = dequant_slab<2, PAIR>(frags, n_have, lane, tmem_a, bar_pempty + 8 * ps, ae, af, parity, abort_flag);
                else if (bits == 3) ok = dequant_slab<3, PAIR>(frags, n_have, lane, tmem_a, bar_pempty + 8 * ps, ae, af, parity, abort_flag);
                else ok = dequant_slab<4, PAIR>(frags, n_have, lane, tmem_a, bar_pempty + 8 * ps, ae, af, parity, abort_flag);
            }
        }
    } else if (warp < GM_TMA) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(GM_REGS_EP));
        // ---------------- epilogue: TMEM lane quarter (warp & 3) -> out[token][row] -------------------------------
        const int quarter = warp & 3;
        const uint32_t dempty = PAIR ? cluster_map(bar_dempty, 0) : bar_dempty;
        float* stg = reinterpret_cast<float*>(sC + quarter * T::CHUNKS * 4096);
        uint32_t segc = 0, n_chunks = 0;
        bool ok = true;
        while (ok && gemm_next_seg<PAIR>(pos, run_hi, a, rank, sg)) {
            const GemmOp& op = a.op[sg.op];
            const uint32_t buf = n_buf == 2 ? (segc & 1u) : 0u, use = n_buf == 2 ? (segc >> 1) : segc;
            ++segc;
            pdl_wait();   // scales, outputs and tile flags belong to the stream's order (returns at once after the first time)
            // token rows whose input was divided by a power of two get it back below (rare): asked while the sums are built
            bool scaled = false;
            if (a.tok_scale != nullptr) {
#pragma unroll
                for (int i = 0; i < T::MAX_TN / 32; ++i) scaled |= __ldcg(a.tok_scale + min(sg.st * a.tn + 32 * i + lane, a.M - 1)) != 1.f;
                scaled = __any_sync(0xffffffffu, scaled);
            }
            ok = mbar_wait_warp<PAIR>(bar_dfull + 8 * buf, use & 1, abort_flag, 7);
            if (!ok) break;
            tc_fence_after();
            // with a residual the launcher has copied it into out: every run then adds on top of it
            const bool first_mode = a.store_first && op.res == nullptr;
            const bool entire = (sg.s0 == 0 && sg.s1 == a.n_slabs);
            const bool whole = (entire && (op.res == nullptr || !a.tma_out)) || (first_mode && sg.s1 == a.n_slabs);
            const bool raise_flag = first_mode && whole && !entire;
            if (first_mode && !whole) {   // the tile's last-slab run has to have stored before anything is added
                const uint32_t* fl = &g_tile_flags[a.flag_slot][sg.tile][rank * GM_EP_WARPS + quarter];
                uint32_t seen = 0, spins = 0;
                if (lane == 0) {
                    while ((seen = ld_acquire_u32(fl)) != a.epoch) {
                        if (++spins > (1u << 22) || *abort_flag) break;
                        __nanosleep(100);
                    }
                    if (seen != a.epoch) give_up<PAIR>(abort_flag, 8);
                    asm volatile("fence.proxy.async;" ::: "memory");   // (the additions below go through the asynchronous proxy)
                }
                seen = __shfl_sync(0xffffffffu, seen, 0);
                ok = (seen == a.epoch);
                if (!ok) break;
            }
            const bool add_res = (op.res != nullptr && sg.s0 == 0 && !a.tma_out);
            const CUtensorMap* tmo = &tmap_out.m[sg.op];
            const int tok0 = sg.st * a.tn, halves = PAIR ? (sg.n_rt > 0 ? 1 : 0) : sg.n_rt > 8 ? 2 : 1;
            const uint32_t td = tmem_base + buf * 128u + ((uint32_t)(quarter * 32) << 16);
            const int n_cc = (sg.w + 31) / 32, n_all = halves * n_cc;
            auto column = [&](int c) -> uint32_t { const int rh = c >= n_cc ? 1 : 0; return td + (uint32_t)(rh * d_cols + (c - rh * n_cc) * 32); };
            auto emit = [&](uint32_t (&v)[32], int c) {
#pragma unroll
                for (int j = 0; j < 32; ++j) asm volatile("" : "+r"(v[j]));   // (read only after the wait)
                const int rh = c >= n_cc ? 1 : 0, c0 = (c - rh * n_cc) * 32, n0 = sg.rt * GM_ROWS + (PAIR ? rank : rh) * 128 + quarter * 32;
                if (scaled) {
                    const float sc = __ldcg(a.tok_scale + min(tok0 + c0 + lane, a.M - 1));
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * __shfl_sync(0xffffffffu, sc, j));
                }
                if (a.tma_out) {
                    if (lane == 0) bulk_wait_read<T::CHUNKS - 1>();   // the copy that last read this chunk has left shared memory
                    __syncwarp();
                    float* chunk = stg + (n_chunks++ % T::CHUNKS) * 1024;      // [32 tokens][32 rows]
#pragma unroll
                    for (int j = 0; j < 32; ++j) chunk[j * 32 + lane] = __uint_as_float(v[j]);
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) {   // rows / tokens past the end of the tensor are clipped by the copy
                        if (whole) tma_store_2d(tmo, smem_u32(chunk), n0, tok0 + c0);
                        else tma_reduce_add_2d(tmo, smem_u32(chunk), n0, tok0 + c0);
                        bulk_commit();
                    }
                } else {
                    const int64_t n = (int64_t)n0 + lane;
                    const int left = min(sg.w - c0, a.M - tok0 - c0);   // tokens of the chunk
                    if (n < op.N) {
                        const int64_t at = (int64_t)(tok0 + c0) * op.ldo + n;
                        float* o = op.out + at;
                        if (add_res) {
                            const float* r = op.res + at;
#pragma unroll
                            for (int j = 0; j < 32; ++j, r += op.ldo)
                                if (j < left) v[j] = __float_as_uint(__uint_as_float(v[j]) + __ldg(r));
                        }
                        if (whole) {
#pragma unroll
                            for (int j = 0; j < 32; ++j, o += op.ldo)
                                if (j < left) *o = __uint_as_float(v[j]);
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j, o += op.ldo)
                                if (j < left) atomicAdd(o, __uint_as_float(v[j]));
                        }
                    }
                }
            };
            // two register sets: the TMEM load of the next 32 columns is in flight while this one is staged
            uint32_t va[32], vb[32];
            if (!PAIR || n_all > 0) tmem_ld32(column(0), va);
            for (int c = 0; c < n_all; c += 2) {
                tmem_ld_wait();
                if (c + 1 < n_all) tmem_ld32(column(c + 1), vb);
                emit(va, c);
                if (c + 1 < n_all) {
                    tmem_ld_wait();
                    if (c + 2 < n_all) tmem_ld32(column(c + 2), va);
                    emit(vb, c + 1);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_issuer<PAIR>(dempty + 8 * buf);   // the next instructions may overwrite the accumulators
            if (raise_flag) {
                if (lane == 0) {
                    bulk_wait_all<0>();   // this warp's stores must have landed before its flag goes up
                    asm volatile("fence.proxy.async;" ::: "memory");
                    if (!a.hold) st_release_u32(&g_tile_flags[a.flag_slot][sg.tile][rank * GM_EP_WARPS + quarter], a.epoch);
                }
                __syncwarp();
            }
        }
        if (lane == 0) bulk_wait_all<0>();   // this thread's output copies are complete
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(GM_REGS_OTHER));
    if (warp == GM_TMA) {
        // ---------------- producer: token tiles (TMA) ---------------------------------------------
        if (lane == 0) {
            uint32_t bi = 0;
            bool ok = true;
            const uint32_t bfull = PAIR ? cluster_map(bar_bfull, 0) : bar_bfull;
            pdl_wait();   // x is the predecessor's output
            while (ok && gemm_next_seg<PAIR>(pos, run_hi, a, rank, sg)) {
                for (int it = 2 * sg.s0; it < 2 * sg.s1 && ok; ++it) {
                    const uint32_t bs = bi % T::B_SLOTS;
                    ok = mbar_wait<PAIR>(bar_bempty + 8 * bs, ((bi / T::B_SLOTS) & 1) ^ 1, abort_flag, 2);
                    if (!ok) break;
                    if (rank == 0) mbar_expect_tx(bar_bfull + 8 * bs, (uint32_t)(a.tn * 128));
                    if constexpr (PAIR) tma_load_2d_pair(smem_u32(sB + bs * T::B_BYTES), &tmap_x, it * GM_KSTAGE, sg.st * a.tn + rank * (sg.w / 2), bfull + 8 * bs);
                    else tma_load_2d(smem_u32(sB + bs * T::B_BYTES), &tmap_x, it * GM_KSTAGE, sg.st * a.tn, bfull + 8 * bs);
                    ++bi;
                }
            }
        }
        __syncwarp();
    } else if (warp == GM_PACKED) {
        // ---------------- producer: packed fragments (bulk copies) ----------------------------------
        if (lane == 0) {
            uint32_t pi = 0;
            bool ok = true;
            while (ok && gemm_next_seg<PAIR>(pos, run_hi, a, rank, sg)) {
                const GemmOp& op = a.op[sg.op];
                const int FB = frag_bytes(op.bits);
                for (int s = sg.s0; s < sg.s1; ++s) {
                    const uint32_t ps = pi % GM_PSTAGES;
                    ok = mbar_wait<PAIR, true>(bar_pempty + 8 * ps, ((pi / GM_PSTAGES) & 1) ^ 1, abort_flag, 1);
                    if (!ok) break;
                    mbar_expect_tx(bar_pfull + 8 * ps, (uint32_t)(sg.n_rt * FB));
                    if (!PAIR || sg.n_rt > 0) bulk_load(smem_u32(sP + ps * T::P_BYTES), op.frags + frag_index(s, sg.rt * GM_FRAGS + rank * T::FRAGS, op.NT) * FB, (uint32_t)(sg.n_rt * FB), bar_pfull + 8 * ps);
                    ++pi;
                }
            }
        }
        __syncwarp();
    } else if (warp == GM_MMA) {
        // ---------------- MMA issue ----------------------------------------------------------------
        uint32_t ai = 0, bi = 0, segc = 0;
        bool ok = rank == 0;
        while (ok && gemm_next_seg<PAIR>(pos, run_hi, a, rank, sg)) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(sg.w >> 3) << 17) | ((PAIR ? 16u : 8u) << 24);   // f16 x f16 -> f32, 128 (a pair: 256) x w
            const uint32_t buf = n_buf == 2 ? (segc & 1u) : 0u, use = n_buf == 2 ? (segc >> 1) : segc;
            ++segc;
            ok = mbar_wait_warp<PAIR>(bar_dempty + 8 * buf, (use & 1) ^ 1, abort_flag, 9);
            if (!ok) break;
            tc_fence_after();
            const uint32_t td = __shfl_sync(0xffffffffu, tmem_base + buf * 128u, 0);
            const bool both = sg.n_rt > 8;
            for (int it = 2 * sg.s0; it < 2 * sg.s1 && ok; ++it) {
                const uint32_t as = ai % T::A_STAGES, bs = bi % T::B_SLOTS;
                ok = mbar_wait_warp<PAIR>(bar_afull + 8 * as, (ai / T::A_STAGES) & 1, abort_flag, 3) && mbar_wait_warp<PAIR>(bar_bfull + 8 * bs, (bi / T::B_SLOTS) & 1, abort_flag, 4);
                if (!ok) break;
                tc_fence_after();
                const uint64_t bd = make_smem_desc(__shfl_sync(0xffffffffu, smem_u32(sB) + bs * T::B_BYTES, 0));
                const uint32_t ta = __shfl_sync(0xffffffffu, tmem_base + GM_ACOL0 + as * T::A_COLS, 0);
                const uint32_t more = it > 2 * sg.s0 ? 1u : 0u;
                if (elect_one()) {
#pragma unroll
                    for (int k = 0; k < GM_KSTAGE / 16; ++k) {
                        if constexpr (PAIR) umma_f16_ts_pair(td, ta + 8 * k, bd + 2 * k, idesc, k > 0 ? 1u : more);
                        else umma_f16_ts(td, ta + 8 * k, bd + 2 * k, idesc, k > 0 ? 1u : more);
                        if (!PAIR && both) umma_f16_ts(td + d_cols, ta + 32 + 8 * k, bd + 2 * k, idesc, k > 0 ? 1u : more);
                    }
                    commit_all<PAIR>(bar_bempty + 8 * bs);
                    commit_all<PAIR>(bar_aempty + 8 * as);
                    if (it + 1 == 2 * sg.s1) commit_all<PAIR>(bar_dfull + 8 * buf);
                }
                __syncwarp();
                ++ai; ++bi;
            }
        }
    }
    }
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) __nanosleep(200000);   // let copies in flight land before the CTA's shared memory goes away
    __syncwarp();
    if constexpr (PAIR) cluster_sync_all();  // neither CTA leaves, or frees its TMEM, while the other's barriers, copies or instructions reach into it
    if (warp == GM_TMA) {
        tc_fence_after();
        if constexpr (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(512) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "n"(512) : "memory");
    }
}

// ---- host ---------------------------------------------------------------------
EncodeTiledFn tensor_map_encoder() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess &&
            qr == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

template <bool PAIR>
static cudaError_t launch_one(const CUtensorMap& tm, const GemmOutMaps& tmo, const GemmArgs& a, int workers, cudaStream_t s) {
    auto kern = gemm_kernel<PAIR>;
    static PerDeviceOnce configured;
    {
        const int rc = configured.run(current_device(), [&] {
            return (int)cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Tile<PAIR>::SMEM);
        });
        if (rc != 0) return rc < 0 ? cudaErrorInvalidDevice : (cudaError_t)rc;
    }
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)(PAIR ? 2 * workers : workers)); cfg.blockDim = dim3(GM_THREADS); cfg.dynamicSmemBytes = Tile<PAIR>::SMEM; cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = 2; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = PAIR ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, tm, tmo, a);
    count_launch();
    return e;
}

static GemmShape shape_of(const aq_handle_s* const* hs, int n, int M) {
    long long R = 0;
    for (int i = 0; i < n; ++i) R += (hs[i]->NT + GM_FRAGS - 1) / GM_FRAGS;
    return gemm_shape(R, hs[0]->KP, M, sm_count());
}

// cut_runs for tiles of c1 units, remembered: finding the runs takes the host about 10 us, a stack asks for the same few
// partitions again and again.
static void cached_runs(long long total, long long c1, int grid, int seg_cost, int* bounds) {
    struct Entry { long long total, c1; int grid, seg_cost; int bounds[GM_MAX_GRID + 1]; };
    static std::mutex m;
    static std::vector<Entry> entries;   // (at most 64: the oldest makes room)
    std::lock_guard<std::mutex> lock(m);
    for (const Entry& e : entries)
        if (e.total == total && e.c1 == c1 && e.grid == grid && e.seg_cost == seg_cost) { memcpy(bounds, e.bounds, sizeof(e.bounds)); return; }
    Entry e;
    memset(&e, 0, sizeof(e));
    e.total = total; e.c1 = c1; e.grid = grid; e.seg_cost = seg_cost;
    cut_runs(total, c1, grid, e.bounds, seg_cost);
    memcpy(bounds, e.bounds, sizeof(e.bounds));
    if (entries.size() >= 64) entries.erase(entries.begin());
    entries.push_back(e);
}

// n (<= GM_MAX_OPS) matrices with the same K against one x: out[i] = (res[i]) + x W_i^T.
// outs_ready: the caller has already put the residual (or zeros) into every output.
cudaError_t launch_gemm_group(const aq_handle_s* const* hs, int n, const void* x16, const float* tok_scale, int M, float* const* outs,
                              const int64_t* ldos, const float* const* ress, bool outs_ready, cudaStream_t s) {
    EncodeTiledFn enc = tensor_map_encoder();
    if (!enc || n < 1 || n > GM_MAX_OPS) return cudaErrorNotSupported;
    GemmArgs a;
    memset(&a, 0, sizeof(a));
    a.n_ops = n; a.M = M; a.n_slabs = hs[0]->KP * 2;
    a.tok_scale = tok_scale;
    long long rows = 0;
    for (int i = 0; i < n; ++i) {
        if (hs[i]->K != hs[0]->K) return cudaErrorInvalidValue;
        GemmOp& o = a.op[i];
        o.frags = hs[i]->frags; o.out = outs[i]; o.res = ress ? ress[i] : nullptr; o.ldo = ldos[i];
        o.N = (int)hs[i]->N; o.NT = hs[i]->NT; o.R = (hs[i]->NT + GM_FRAGS - 1) / GM_FRAGS; o.bits = hs[i]->bits;
        rows += o.R;
    }
    const GemmShape shape = shape_of(hs, n, M);
    a.n_st = shape.n_st; a.tn = shape.tn;
    const long long tiles = rows * a.n_st, total = tiles * 2 * a.n_slabs;   // in half slabs
    int grid = shape.workers;
    if (total / 2 < grid) grid = (int)(total / 2);
    if (total > 0x7fffffffLL) return cudaErrorInvalidValue;
    cached_runs(total, 2LL * a.n_slabs, grid, shape.pair ? GM_PAIR_SEG_COST : GM_SEG_COST, a.bounds);
    CUtensorMap tm;
    const cuuint64_t dims[2] = {(cuuint64_t)hs[0]->K, (cuuint64_t)M};
    const cuuint64_t strides[1] = {(cuuint64_t)hs[0]->K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)GM_KSTAGE, (cuuint32_t)(shape.pair ? a.tn / 2 : a.tn)};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(&tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void*>(x16), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    // the outputs as tensors [M][N] of float32 for the epilogue's 32 x 32 copies (row pitch must be 16-byte aligned)
    GemmOutMaps tmo;
    memset(&tmo, 0, sizeof(tmo));
    a.tma_out = 1;
    for (int i = 0; i < n && a.tma_out; ++i) {
        const GemmOp& o = a.op[i];
        if (o.ldo % 4 != 0 || (reinterpret_cast<uintptr_t>(o.out) & 15u) != 0) { a.tma_out = 0; break; }
        const cuuint64_t odims[2] = {(cuuint64_t)o.N, (cuuint64_t)M};
        const cuuint64_t ostrides[1] = {(cuuint64_t)o.ldo * 4};
        const cuuint32_t obox[2] = {32, 32};
        if (enc(&tmo.m[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, o.out, odims, ostrides, obox, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            a.tma_out = 0;
    }
    // What an output holds before the kernel: the residual when there is one (every run then adds to it);
    // else zeros when some run does not cover a whole tile; else nothing.
    bool all_whole = true;
    {
        for (int c = 1; c < grid && all_whole; ++c) all_whole = a.bounds[c] % (2 * a.n_slabs) == 0;
    }
    if (outs_ready && !a.tma_out) return cudaErrorInvalidValue;   // (the caller checks gemm_outputs_can_be_preset first)
    static std::atomic<uint32_t> epoch_counter{0};
    a.store_first = (a.tma_out && gemm_stores_first(hs, n, M, s)) ? 1 : 0;
    a.epoch = epoch_counter.fetch_add(1) + 1;
    if (a.epoch == 0) a.epoch = epoch_counter.fetch_add(1) + 1;   // flags start out as zero: never use that value
    a.flag_slot = (int)(a.epoch % GM_FLAG_SLOTS);
    a.hold = g_gemm_hold.load(std::memory_order_relaxed) ? 1 : 0;
    // What an output holds before the kernel: the residual when there is one (every run then adds to it); zeros
    // when runs add without the store-first protocol; else nothing.  With outs_ready the caller has done this.
    for (int i = 0; i < n && !outs_ready; ++i) {
        const GemmOp& o = a.op[i];
        cudaError_t e = cudaSuccess;
        if (o.res && a.tma_out)
            e = cudaMemcpy2DAsync(o.out, (size_t)o.ldo * sizeof(float), o.res, (size_t)o.ldo * sizeof(float),
                                  (size_t)o.N * sizeof(float), (size_t)M, cudaMemcpyDeviceToDevice, s);
        else if (!all_whole && !(a.store_first && !o.res))
            e = cudaMemset2DAsync(o.out, (size_t)o.ldo * sizeof(float), 0, (size_t)o.N * sizeof(float), (size_t)M, s);
        if (e != cudaSuccess) return e;
    }
    return shape.pair ? launch_one<true>(tm, tmo, a, grid, s) : launch_one<false>(tm, tmo, a, grid, s);
}

cudaError_t launch_gemm(const aq_handle_s* h, const void* x16, const float* tok_scale, int M, float* out, int64_t ldo, bool out_ready, cudaStream_t s) {
    const float* res = nullptr;
    return launch_gemm_group(&h, 1, x16, tok_scale, M, &out, &ldo, &res, out_ready, s);
}

// ---- activations -> the operand ---------------------------------------------------------------------------------------
// Binary16 rows in operand order (operand_position).  One CTA per token row.  A bfloat16 value has 8 significant bits, so it
// is a binary16 value whenever it is inside binary16's range (magnitudes below 2^-17 land on the subnormal grid, an absolute
// error below 2^-25).  A row that holds a magnitude of 2^15 or more is divided by the power of two that brings its largest one
// below 2^15 (exact for everything that stays normal); scale[m] is that power of two, 1 otherwise.  Binary16 rows are only
// reordered (scale unused).  zero (or null): rows of zero4 groups of four floats that the GEMM will add to.
template <bool BF16>
__global__ void __launch_bounds__(256) operand_rows_kernel(const uint16_t* __restrict__ x, __half* __restrict__ x16,
                                                           float* __restrict__ scale, int64_t K, float4* __restrict__ zero, int64_t zero4) {
    const int64_t m = blockIdx.x;
    pdl_wait();
    const uint16_t* xr = x + m * K;
    __half* o = x16 + m * K;
    pdl_launch_dependents();
    const int q8 = (int)(K >> 3), wid = (int)threadIdx.x & ~31;   // groups of eight elements (K is a multiple of 32); the warp's first thread
    float mx = 0.f;
    auto convert = [&](uint4& v, float f, bool on) {   // bfloat16 -> binary16, times f
        uint32_t* w = reinterpret_cast<uint32_t*>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 p = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(w + i));
            const __half2 h = __floats2half2_rn(p.x * f, p.y * f);
            w[i] = *reinterpret_cast<const uint32_t*>(&h);
            if (on) mx = fmaxf(mx, fmaxf(fabsf(p.x), fabsf(p.y)));
        }
    };
    auto rows = [&](float f) {
        constexpr int STEPS = 4;   // groups per thread whose loads go out together
        for (int i0 = 0; i0 + wid < q8; i0 += 256 * STEPS) {
            uint4 v[STEPS];
#pragma unroll
            for (int n = 0; n < STEPS; ++n) {
                const int i = i0 + 256 * n + (int)threadIdx.x;
                v[n] = i < q8 ? *reinterpret_cast<const uint4*>(xr + 8 * (int64_t)i) : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int n = 0; n < STEPS; ++n) {
                const int i = i0 + 256 * n + (int)threadIdx.x;
                if (i0 + 256 * n + wid >= q8) break;
                if constexpr (BF16) convert(v[n], f, i < q8);
                store_operand8(o, 8 * (int64_t)i, v[n], i < q8);
            }
        }
    };
    rows(1.f);
    for (int64_t i = threadIdx.x; i < zero4; i += 256) zero[m * zero4 + i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (BF16) {
        __shared__ float red[8];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
        __syncthreads();
        mx = red[0];
#pragma unroll
        for (int i = 1; i < 8; ++i) mx = fmaxf(mx, red[i]);
        float sc = 1.f;
        if (mx >= 32768.f && mx <= 3.0e38f) {   // (non-finite input stays non-finite: nothing to rescue)
            int e;
            frexpf(mx, &e);                       // mx = f 2^e, f in [0.5, 1)
            sc = ldexpf(1.f, e - 15);             // mx / sc in [2^14, 2^15)
            rows(1.f / sc);
        }
        if (threadIdx.x == 0) scale[m] = sc;
    }
}

cudaError_t launch_operand_rows(const void* x, aq_dtype_t dt, void* x16, float* scale, int M, int64_t K, float* zero, int64_t zero_width, cudaStream_t s) {
    const uint16_t* xu = reinterpret_cast<const uint16_t*>(x);
    __half* o = reinterpret_cast<__half*>(x16);
    const cudaError_t e = launch_pdl(dt == AQ_BF16 ? operand_rows_kernel<true> : operand_rows_kernel<false>, dim3((unsigned)M), dim3(256), 0, s, xu, o, scale, K,
                                     reinterpret_cast<float4*>(zero), zero ? zero_width / 4 : (int64_t)0);
    count_launch();
    return e;
}

// True when outputs without a residual need no zeroing before launch_gemm_group (split tiles store first).
bool gemm_stores_first(const aq_handle_s* const* hs, int n, int M, cudaStream_t s) {
    // The protocol tells launches apart by a fresh epoch per launch.  A launch recorded into a CUDA graph would run
    // again with the epoch it was recorded with, so while a stream is being captured outputs are zeroed and added to.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) { cudaGetLastError(); return false; }
    if (cap != cudaStreamCaptureStatusNone) return false;
    // Stores first saves writing the zeros, but where a tile is shared by CTAs that all reach it at the same time the others
    // wait 3 to 5 us for the first one's stores; from about two CTAs per tile on, zeros are cheaper.  Measured, stores first /
    // zeros: 4096 x 4096 (16 tiles) at 32 tokens 18.5 / 15.2 us, 11008 x 4096 (86 tiles) at 200 tokens 46 / 42 us, eight 7B
    // layers (48 and 86 tiles) at 50 tokens 814 / 739 us; the other way round with 104 to 148 tiles, 18 expert layers at 512
    // tokens 1291 / 1381 us.  On pairs (74, so from 52 tiles on): 44 tiles (2688 x 8192 at 1024 tokens) 55.9 / 52.5 us, 48 (4096 x
    // 4096 at 768) 37.1 / 33.7; 60 (5003 x 4000 at 768) 39.4 / 42.0, 64 (4096 x 4096 at 1024) 40.2 / 41.4, but with twice the columns
    // 75.5 / 72.0, 86 (11008 x 4096 at 512) 52.2 / 54.6.
    const GemmShape shape = shape_of(hs, n, M);
    const long long tiles = shape.tiles;
    return tiles <= GM_MAX_TILES && 10 * tiles >= 7 * shape.workers;
}

// True when launch_gemm_group accepts outputs preset by the caller (they are written through tensor maps).
bool gemm_outputs_can_be_preset(float* const* outs, const int64_t* ldos, int n) {
    if (!tensor_map_encoder()) return false;
    for (int i = 0; i < n; ++i)
        if (ldos[i] % 4 != 0 || (reinterpret_cast<uintptr_t>(outs[i]) & 15u) != 0) return false;
    return true;
}

void set_gemm_hold(bool on) { g_gemm_hold.store(on, std::memory_order_relaxed); }

int read_gemm_status(bool clear) {
    int v = 0;
    cudaMemcpyFromSymbol(&v, g_gemm_status, sizeof(int));
    if (clear && v) { int z = 0; cudaMemcpyToSymbol(g_gemm_status, &z, sizeof(int)); }
    return v;
}

}  // namespace aq
