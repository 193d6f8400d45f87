"""Host logic of the prefill GEMM's scheduler: `csrc/aq_gemm_runs.h` (how the (row tile, token tile, half k-slab)
work is cut into one contiguous run per CTA or pair of CTAs), compiled with the host compiler alone and driven from a
small C++ program.  Checked for many shapes, for CTAs and for pairs: the bounds partition the work (ascending, even, first 0, last total), the run that
holds a tile's last slab starts inside that tile or covers the tile whole (what the store-first protocol of the kernel
relies on), and the most expensive run is never more expensive than under the equal cut it replaced."""
import os
import shutil
import subprocess
import textwrap

import pytest

from gemm_rule import gemm_shape

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_2605_24011_b200", "csrc")

SRC = textwrap.dedent(r"""
    #include <algorithm>
    #include <cstdio>
    #include <vector>
    #include "aq_gemm_runs.h"
    using namespace aq;
    #define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s (n_slabs %lld R %lld M %d grid %d)\n", __LINE__, #c, n_slabs, R, M, grid); return 1; } } while (0)

    // the launcher's tiles: 256 rows x up to 128 tokens for a CTA, 256 for a pair; work in half slabs
    static int one(long long n_slabs, long long R, int M, int grid, bool pair) {
        const int tokens = pair ? GM_PAIR_TOKENS : GM_TOKENS, seg = pair ? GM_PAIR_SEG_COST : GM_SEG_COST;
        if (pair) grid /= 2;
        const long long n_st = (M + tokens - 1) / tokens, c1 = 2 * n_slabs, total = R * n_st * c1;
        if (total / 2 < grid) grid = (int)(total / 2);
        if (grid < 1) return 0;
        std::vector<int> b(grid + 1, -1);
        cut_runs(total, c1, grid, b.data(), seg);
        CHECK(b[0] == 0 && b[grid] == total);
        long long worst = 0;
        for (int c = 0; c < grid; ++c) {
            CHECK(b[c] <= b[c + 1] && b[c] % 2 == 0);
            worst = std::max(worst, run_cost(b[c], b[c + 1], c1, seg));
        }
        // a run that contains a tile's last unit and does not start inside that tile covers the tile whole
        for (int c = 0; c < grid; ++c) {
            for (long long pos = b[c]; pos < b[c + 1];) {
                const long long ts = pos / c1 * c1, te = ts + c1;
                if (te <= b[c + 1] && ts < b[c]) CHECK(pos == b[c]);          // the tile's tail: first thing of the run
                pos = std::min<long long>(te, b[c + 1]);
            }
        }
        // never worse than equal runs
        long long worst_equal = 0;
        for (int c = 0; c < grid; ++c) {
            const long long lo = (total * c / grid) & ~1LL, hi = (c + 1 == grid) ? total : ((total * (c + 1) / grid) & ~1LL);
            worst_equal = std::max(worst_equal, run_cost(lo, hi, c1, seg));
        }
        CHECK(worst <= worst_equal);
        // and no run costs more than the work spread evenly plus what one tile and its pieces can add
        CHECK(worst <= total / grid + c1 + 4 * seg + 2 || worst <= worst_equal);
        return 0;
    }

    int main() {
        const int Ms[] = {9, 16, 50, 130, 200, 256, 257, 300, 512, 513, 768, 1000, 1024, 4096};
        const long long Ks[] = {256, 1024, 4096, 11008, 16384};
        const long long Ns[] = {16, 128, 1000, 1024, 2048, 4096, 11008, 12288, 22016, 65536};
        const int grids[] = {1, 7, 132, 148, 160, 192};
        int n = 0;
        for (int M : Ms) for (long long K : Ks) for (long long N : Ns) for (int g : grids) {
            const long long n_slabs = (K + 255) / 256 * 2, R = (N + 255) / 256;
            if (n_slabs * R * 16 > 2000000000LL) continue;
            for (bool pair : {false, true}) {
                if (one(n_slabs, R, M, g, pair)) return 1;
                ++n;
            }
        }
        std::printf("OK %d\n", n);
        return 0;
    }
""")

@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
@pytest.mark.parametrize("pair,N,K,M,sms", [
    (1, 22016, 4096, 512, 148), (1, 22016, 4096, 385, 148), (0, 22016, 4096, 384, 148), (0, 22016, 4096, 640, 148), (1, 4096, 4096, 1024, 148),
    (0, 4096, 4096, 512, 148), (0, 22016, 4096, 512, 1),
    (0, 512, 65536, 448, 148), (0, 128, 131072, 400, 148), (0, 768, 32768, 768, 148), (1, 1024, 16384, 1024, 148),      # few row tiles
    (0, 65536, 256, 1024, 148), (0, 32768, 1024, 512, 148), (1, 32768, 1280, 512, 148),                                  # short rows
    (0, 2048, 16384, 2048, 148), (0, 3072, 16384, 2048, 148), (1, 2304, 16384, 2048, 148), (1, 2304, 8192, 4096, 148),   # 64 MB of tokens
    (1, 4096, 11008, 4096, 148), (1, 11008, 4096, 8192, 148),
])
def test_pairs_where_they_pay(tmp_path, pair, N, K, M, sms):
    got, n_st, tn, workers, tiles = gemm_shape(tmp_path, N, K, M, sms)
    assert got == pair and workers == (sms // 2 if pair else sms) and tiles == n_st * -(-N // 256)
    assert tn <= (256 if pair else 128) and tn % 32 == 0 and (n_st - 1) * tn < M <= n_st * tn


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_gemm_runs_partition(tmp_path):
    src = tmp_path / "runs.cpp"
    exe = tmp_path / "runs"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", HDR, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("OK")
