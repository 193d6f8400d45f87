// Host-only: how the prefill GEMM's work is cut into one contiguous run per CTA.  Plain C++ (no CUDA), so that the
// partition can be tested with the host compiler alone.
#pragma once
#include <cstdint>

namespace aq {

constexpr int GM_MAX_GRID = 192;   // CTAs of one launch (one per SM)
// What ending one piece of a tile costs a CTA (accumulators drained, epilogue, adds of a shared tile), in half slabs of 64 k:
// the runs are cut so that work + pieces balance.  Set by time: over 90 shapes of 9 to 1024 tokens, against 9, a cost of 1
// takes 1.03 to 1.04 of the time, 2 1.01 to 1.04, 3 1.00 to 1.02, 4 to 14 0.99 to 1.015; eight 7B layers at 200 tokens 1191,
// 1156, 1139, 1136, 1133 (6), 1131 (9), 1135 us (14).
constexpr int GM_SEG_COST = 9;
// The same for a CTA pair, whose tiles are twice as wide: of 5, 9 and 15, in us, 4096 x 4096 at 1024 tokens 41.0, 42.1, 37.7,
// 11008 x 4096 at 512 48.9, 46.1, 46.1, 12288 x 4096 52.9, 49.9, 49.8, 22016 x 4096 79.2, 79.1, 79.2.
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
inline long long run_cost(long long lo, long long hi, long long c1) {
    long long cost = 0;
    for (long long pos = lo; pos < hi;) {
        const long long te = (pos / c1 + 1) * c1, end = te < hi ? te : hi;
        cost += GM_SEG_COST + (end - pos);
        pos = end;
    }
    return cost;
}

}  // namespace aq
