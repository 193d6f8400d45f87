"""The prefill GEMM's rule for CTAs or pairs of them, asked of `csrc/aq_gemm_runs.h` through the host compiler."""
import os
import subprocess
import textwrap

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_24011_b200", "csrc")
SRC = textwrap.dedent(r"""
    #include <cstdio>
    #include "aq_gemm_runs.h"
    int main() {
        long long N, K; int M, sms;
        if (std::scanf("%lld %lld %d %d", &N, &K, &M, &sms) != 4) return 1;
        const aq::GemmShape g = aq::gemm_shape((N + 255) / 256, (int)((K + 255) / 256), M, sms);
        std::printf("%d %d %d %d %lld\n", g.pair, g.n_st, g.tn, g.workers, g.tiles);
    }
""")


def gemm_shape(tmp_path, N, K, M, sms):
    """(pairs?, token tiles, tokens per tile, CTAs or pairs, tiles) of one N x K matrix at M tokens on a device of that many SMs."""
    src, exe = tmp_path / "shape.cpp", tmp_path / "shape"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", HDR, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], input=f"{N} {K} {M} {sms}", capture_output=True, text=True, check=True)
    return tuple(map(int, r.stdout.split()))
