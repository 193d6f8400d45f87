"""The lengths of the decode kernel's rings: `csrc/aq_decode_rings.h` compiled with the host compiler alone.  For every small choice
of lengths the waits of the kernel's roles are written down as an order of events, and whatever `ds_rings_hold` accepts has to be
sound in it: no slot is written before its last unit is through with it, and no wait on a barrier's parity starts a phase too early
or ends a phase too late."""
import os
import shutil
import subprocess
import textwrap

import pytest

HDR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_24011_b200", "csrc")

SRC = textwrap.dedent(r"""
    #include <cstdio>
    #include <vector>
    #include "aq_decode_rings.h"
    using namespace aq;
    constexpr int N = 24;                                   // units
    struct Order {                                          // before[x] holds y: event y has happened whenever x has
        std::vector<std::vector<char>> before;
        int U(int n) { return n; }                          // unpacked: operand, descriptor and scales stored
        int I(int n) { return N + n; }                      // instructions issued
        int F(int n) { return 2 * N + n; }                  // instructions completed
        int C(int n) { return 3 * N + n; }                  // sums, descriptor and scales read
        Order() : before(4 * N, std::vector<char>(4 * N, 0)) {}
        void after(int x, int y) { before[x][y] = 1; }
        void close() {
            for (int k = 0; k < 4 * N; ++k) for (int x = 0; x < 4 * N; ++x) if (before[x][k])
                for (int y = 0; y < 4 * N; ++y) before[x][y] |= before[k][y];
        }
        bool has(int x, int y) { return x == y || before[x][y]; }
    };
    static bool sound(int a, int d, int meta, int teams, bool late) {   // late: the operand's stage is filled again after the sums have been read
        Order o;
        for (int n = 0; n < N; ++n) {
            if (n) { o.after(o.U(n), o.U(n - 1)); o.after(o.I(n), o.I(n - 1)); o.after(o.F(n), o.F(n - 1)); }
            if (n >= a) o.after(o.U(n), late ? o.C(n - a) : o.F(n - a));
            if (n >= d) o.after(o.I(n), o.C(n - d));
            if (n >= teams) o.after(o.C(n), o.C(n - teams));
            o.after(o.I(n), o.U(n)); o.after(o.F(n), o.I(n)); o.after(o.C(n), o.F(n));
        }
        o.close();
        // a wait for unit n's phase of a barrier with `slots` phases in flight, by a role whose last event before it is `from` and
        // whose first event behind it is `to`: phase n - slots is over when it starts, phase n + slots is not before it has ended
        auto wait = [&](int n, int slots, int from, int to, auto phase) {
            if (n >= slots && !(from >= 0 && o.has(from, phase(n - slots)))) return false;
            return n + slots >= N || o.has(phase(n + slots), to);
        };
        auto U = [&](int n) { return o.U(n); };
        auto F = [&](int n) { return o.F(n); };
        auto C = [&](int n) { return o.C(n); };
        for (int n = 0; n < N; ++n) {
            if (n + meta < N && !o.has(o.U(n + meta), o.C(n))) return false;          // the slot of what goes with a unit
            const int before_c = n >= teams ? o.C(n - teams) : -1;
            if (!wait(n, meta, n ? o.I(n - 1) : -1, o.I(n), U)) return false;          // issuer: the operand is there
            if (!wait(n, meta, before_c, o.C(n), U)) return false;                     // collect: the same, then
            if (!wait(n, d, o.U(n), o.C(n), F)) return false;                          // ... its instructions
            if (n + a < N && !(late ? wait(n, d, o.U(n + a - 1), o.U(n + a), C) : wait(n, d, o.U(n + a - 1), o.U(n + a), F))) return false;  // unpack
            if (n + d < N && !wait(n, d, o.I(n + d - 1), o.I(n + d), C)) return false;  // issuer: the sums have been read
        }
        return true;
    }
    int main() {
        int accepted = 0;
        for (int teams = 1; teams <= 3; ++teams) for (int a = 1; a <= 4; ++a) for (int d = 1; d <= 4; ++d) for (int m = 1; m <= 8; ++m)
            if (ds_rings_hold(a, d, m, teams)) {
                ++accepted;
                if (!sound(a, d, m, teams, false) || !sound(a, d, m, teams, true)) { std::printf("accepted, but not sound: A %d D %d META %d, %d teams\n", a, d, m, teams); return 1; }
            }
        for (int teams = 2; teams <= 3; ++teams)
            if (!ds_rings_hold(DS_A_STAGES, DS_D_STAGES, DS_META_SLOTS, teams) || sound(2, 2, 3, teams, false)) { std::printf("%d teams\n", teams); return 1; }
        std::printf("OK %d\n", accepted);
        return accepted > 50 ? 0 : 1;
    }
""")


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_decode_rings(tmp_path):
    src, exe = tmp_path / "rings.cpp", tmp_path / "rings"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", HDR, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
