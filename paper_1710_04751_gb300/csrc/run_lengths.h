// run_lengths.h -- which runs of steps lbm_step launches as graphs.  Host only, no CUDA.
#pragma once

#include <stdint.h>

namespace lbm {

// A run of n steps between two checks goes step by step, or as one graph: a program that advances a
// small cavity a few steps at a time spends most of such a call in the launches (24^3, a run of 10
// and one of 20, each waited for: 88 us step by step, 71 as graphs).  Making a graph takes longer
// than many such runs save, so a length gets one when it comes twice in a row while there is room,
// for kSlots lengths; once those are taken, another length displaces the one used less recently when
// it has come kAgain times in a row.  (With room for one length, 10, 10, 20, 20, ... made a graph on
// every second call: 259 us for the four, 143 now.)
struct RunLengths {
    static constexpr int kSlots = 2, kAgain = 16;
    static constexpr int64_t kMin = 4, kMax = 128;
    int64_t len[kSlots] = {0, 0};
    int64_t last = 0;    // the last run's length
    int row = 0;         // and how often it came in a row
    int recent = 0;      // the slot used last
    bool failed = false; // no graph could be made of a run: launch them step by step

    // Counts a run of n steps.  Returns its slot, or -1: step by step.  *replaced: the slot is still
    // free or another length's; the caller drops that one's graphs and calls take().
    int find(int64_t n, bool* replaced) {
        *replaced = false;
        row = n == last ? row + (row < kAgain) : 1;
        last = n;
        if (failed || n < kMin || n > kMax) return -1;
        for (int s = 0; s < kSlots; ++s)
            if (len[s] == n) return recent = s;
        if (row < 2) return -1;
        *replaced = true;
        for (int s = 0; s < kSlots; ++s)
            if (len[s] == 0) return s;
        return row < kAgain ? -1 : (recent + 1) % kSlots;
    }
    void take(int slot, int64_t n) { len[slot] = n, recent = slot; }
};

}  // namespace lbm
