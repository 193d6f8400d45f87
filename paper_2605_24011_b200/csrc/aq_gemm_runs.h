// Host-only: whether the prefill GEMM runs on CTAs or on pairs of them, and how its work is cut into one contiguous run for each.
// Plain C++ (no CUDA), so that rule and partition can be tested with the host compiler alone.
#pragma once
#include <cstdint>

namespace aq {

constexpr int GM_MAX_GRID = 192;   // CTAs of one launch (one per SM)
constexpr int GM_TOKENS = 128, GM_PAIR_TOKENS = 256;   // tokens of a tile at most: of one CTA's, of a pair's

// How a launch is cut: CTAs or pairs of them, token tiles of one width.
struct GemmShape {
    bool pair;
    int n_st, tn;      // token tiles, tokens per tile
    int workers;       // CTAs or pairs that the device holds
    long long tiles;   // of 256 rows x tn tokens
};

// R row tiles of 256 rows, KP x 256 columns, M tokens.
// Pairs dequantise a weight, and read it from L2, once per 256 tokens instead of 128, but fill and drain tiles of twice the size, and a
// tile costs them nearly the same whatever it holds: they pay where the tokens fill tiles of 256 (an even number of 128s, at least
// four) and a pair has about 48 stages (256 rows x 256 tokens x 64 k) of work.  Measured, us with single CTAs / pairs, 3 bits:
// 22016 x 4096 at 256 tokens 47.3 / 46.8, 257 57.9 / 68.5, 384 66.0 / 72.4, 448 82.4 / 75.3, 512 85.7 / 79.7, 640 103.5 / 104.5, 768
// 124.6 / 114.1; 4096 x 11008 at 256 30.5 / 31.3, 512 47.8 / 46.8; 4096 x 4096 at 512 (28 stages) 26.1 / 26.8, at 1024 (55) 43.8 / 37.7.
// Not with less than four row tiles, where twenty pairs and more add to a tile: 512 x 65536 at 512 tokens 58.1 / 61.5, 256 x 65536 at
// 1024 83.2 / 89.7, 768 x 32768 at 768 54.3 / 56.1; 1024 x 16384 at 768 34.6 / 34.1, 1280 x 16384 at 1024 54.9 / 54.4.
// Not for rows of up to 1024, whose tiles end every 16 stages: 65536 x 256 at 1024 159 / 170, 65536 x 512 183 / 189, 32768 x 1024 at 512
// 63.2 / 64.8; 32768 x 1280 at 512 71.1 / 70.6, at 1024 140.5 / 137.6.
// Not for 64 MB of activations and more, where the tokens of the tiles that are worked on at one time come from HBM again, unless the
// pairs go through whole tiles together (nearly whole rounds, or many): 2048 x 16384 at 2048 tokens (64 tiles on 74 pairs) 161 / 167,
// 3072 x 16384 (96) 222 / 235, 4096 x 16384 (128) 304 / 318; 2304 x 16384 (72) 175 / 157, 2304 x 8192 at 4096 (144) 183 / 166, 4096 x
// 11008 at 4096 (256) 424 / 412.
inline GemmShape gemm_shape(long long R, int KP, int M, int sms) {
    GemmShape g;
    if (sms > GM_MAX_GRID) sms = GM_MAX_GRID;
    const int t128 = (M + 127) / 128, pairs = sms / 2;
    g.pair = t128 >= 4 && t128 % 2 == 0 && pairs >= 1 && R * (t128 / 2) * KP * 4 >= 48LL * pairs && R >= 4 && KP > 4;
    if (g.pair && (long long)M * KP * 256 >= 1LL << 25) {
        const long long tiles = R * (t128 / 2), rounds = (tiles + pairs - 1) / pairs;
        g.pair = rounds > 3 || 16 * tiles >= 15 * rounds * pairs;
    }
    g.workers = g.pair ? pairs : sms;
    const int max_tn = g.pair ? GM_PAIR_TOKENS : GM_TOKENS;
    g.n_st = (M + max_tn - 1) / max_tn;
    // (several tiles: a multiple of 32, the width of the epilogue's copies, which must not reach into the next tile; a pair's
    // instruction takes multiples of 32)
    g.tn = g.pair || g.n_st > 1 ? ((M + g.n_st - 1) / g.n_st + 31) / 32 * 32 : (M + 15) / 16 * 16;
    g.tiles = R * g.n_st;
    return g;
}

// What ending one piece of a tile costs a CTA (accumulators drained, epilogue, adds of a shared tile), in half slabs of 64 k:
// the runs are cut so that work + pieces balance.  Set by time: over 90 shapes of 9 to 1024 tokens, against 9, a cost of 1
// takes 1.03 to 1.04 of the time, 2 1.01 to 1.04, 3 1.00 to 1.02, 4 to 14 0.99 to 1.015; eight 7B layers at 200 tokens 1191,
// 1156, 1139, 1136, 1133 (6), 1131 (9), 1135 us (14).
constexpr int GM_SEG_COST = 9;
// The same for a CTA pair, whose tiles are twice as wide: of 5, 9 and 15, in us, 4096 x 4096 at 1024 tokens 41.0, 42.1, 37.7,
// 11008 x 4096 at 512 48.9, 46.1, 46.1, 12288 x 4096 52.9, 49.9, 49.8, 22016 x 4096 79.2, 79.1, 79.2.  Over 75 products that pairs
// take, 400 to 1024 tokens, against 15: 9 takes 1.006 of the time (geometric mean; 0.97 to 1.11), 12 1.002, 21 1.009.
constexpr int GM_PAIR_SEG_COST = 15;

// Cuts [0, total) into `grid` contiguous runs with even bounds (bounds[0] = 0 .. bounds[grid] = total).  The work is a
// sequence of tiles of c1 units each.  A run costs its units plus seg_cost per tile it touches; the smallest budget under
// which a greedy walk places everything is found by bisection.
inline void cut_runs(long long total, long long c1, int grid, int* bounds, int seg_cost = GM_SEG_COST) {
    auto walk = [&](long long budget, int* out) {
        long long pos = 0;
        for (int c = 0; c < grid; ++c) {
            if (out) out[c] = (int)pos;
            long long left = budget;
            while (pos < total) {
                const long long te = (pos / c1 + 1) * c1, need = seg_cost + (te - pos);
                if (need <= left) { pos = te; left -= need; continue; }
                const long long take = (left - seg_cost) & ~1LL;
                if (take >= 2) pos += take;
                break;
            }
        }
        if (out) out[grid] = (int)total;
        return pos >= total;
    };
    long long lo = total / grid, hi = total / grid + 4 * seg_cost + 4;
    while (!walk(hi, nullptr)) hi *= 2;
    while (lo < hi) {
        const long long mid = (lo + hi) / 2;
        if (walk(mid, nullptr)) hi = mid; else lo = mid + 1;
    }
    walk(hi, bounds);   // (a tail of CTAs may be left without work: their runs are empty)
}

// Cost of the run [lo, hi) under the model above.
inline long long run_cost(long long lo, long long hi, long long c1, int seg_cost = GM_SEG_COST) {
    long long cost = 0;
    for (long long pos = lo; pos < hi;) {
        const long long te = (pos / c1 + 1) * c1, end = te < hi ? te : hi;
        cost += seg_cost + (end - pos);
        pos = end;
    }
    return cost;
}

}  // namespace aq
