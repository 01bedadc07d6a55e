// CTAs of a per-thread operation launch.  Host arithmetic alone, compiled
// without CUDA too.
#pragma once

#include <cstdint>

namespace cht {

// The CTAs of overlapping launches go to the SMs that the launch before
// leaves first, so a grid with fewer CTAs than fit crowds on some SMs while
// others idle.  Modifying batches of about one wave run one operation per
// thread (32 rounds of 2^18 inserts and erases behind a growth to 2^24
// cells: 2.45 -> 2.36 ms; a find of that size is 2 % slower so); those with at
// least kThreadOps operations per thread are cut four times finer, so that
// the SMs share them as they come free (counting 2^26 words, then 2^24 finds:
// 2.01 -> 1.57 ms; 2^21 erases on 2^22 cells at load 0.5 62 -> 59 us); between
// the two a finer grid only adds a ragged last wave (2^19 operations: 35.7
// against 37.5 us; 2^20 inserts on 2^24 cells 79 against 82 us).
// A caller who asks for a number of CTAs per SM gets a grid of that many.
constexpr uint64_t kThreadOps = 6;

// need: CTAs of one operation per thread; fit: resident CTAs per SM at most;
// asked: CTAs per SM that the caller wants (0: none); modifies: not a find.
constexpr uint64_t thread_grid(uint64_t need, uint64_t sms, uint64_t fit, int asked, bool modifies) {
    const uint64_t wave = sms * fit;
    uint64_t grid = wave;
    if (asked > 0) {
        if (uint64_t(asked) < fit) grid = sms * uint64_t(asked);
    } else if (modifies && need <= wave + wave / 4) {
        grid = need;
    } else if (need >= wave * kThreadOps) {
        grid = wave * 4;
    }
    if (grid > need) grid = need;
    return grid < 1 ? 1 : grid;
}

}  // namespace cht
