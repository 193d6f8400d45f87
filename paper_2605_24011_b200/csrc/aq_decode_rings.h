// Host-only: the rings through which the several-token decode kernel passes its units on, and what has to hold between their
// lengths.  Plain C++ (no CUDA), so that the condition can be tested with the host compiler alone.
#pragma once

namespace aq {

// Operand stages (A), stages of sums (D), and slots for what goes with a unit: its descriptor, its scales and the barrier that
// says that its operand is there (META).  A is filled again once the instructions have read it (or, later, once the sums have been
// read), D written again once the sums have been read.  Nothing guards a META slot but those two waits: unit n + META is unpacked after the instructions of unit
// n + META - A, which were issued after the sums of unit n + META - A - D had been read, so unit n is through with its slot only
// if META >= A + D.  And a collect warp that waits for unit n's instructions must not be answered by the barrier's phase before:
// unit n was unpacked after the instructions of unit n - A, which come no earlier than those of unit n - D only if A <= D.
constexpr int DS_A_STAGES = 2, DS_D_STAGES = 2, DS_META_SLOTS = 4;
constexpr bool ds_rings_hold(int a, int d, int meta, int teams) { return a >= 1 && a <= d && meta >= a + d && meta >= teams; }

}  // namespace aq
