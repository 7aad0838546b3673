// sw_budgets.h -- how much scratch a call or a plan takes (host).
#pragma once
#include <algorithm>

#include "swgb_internal.h"

namespace swgb {

// Scratch of a call, from its pair count (the only size the host knows without
// reading the device): chunk-boundary rows of the score pass, and for the
// traceback the row checkpoints and the per-warp slots.  A warp's slot is sized
// on the device for its launch's largest part; launches use as many warps as
// fit, and the checkpoints' blocks double until those fit.
constexpr int64_t kScoreBndMin = (int64_t)32 << 20, kScoreBndMax = (int64_t)1 << 30, kScoreBndPerPair = 1024;
// What a call takes for its traceback, and the least that it takes on a card that
// has no more.  Short reads need a tenth of it; 60,000 reads of 1,500 bases take
// 40.7 ms with 160 KB a pair, 42.9 with 64, 55.8 with 24; a fifth of them across
// an intron and a third without a true window 57, 132 and 262 ms.
constexpr int64_t kTbMin = (int64_t)256 << 20, kTbPerPair = (int64_t)160 << 10;
constexpr int64_t kTbLeastMin = (int64_t)64 << 20, kTbLeastPerPair = (int64_t)32 << 10;
// Bounds of a stream's largest traceback scratch, and its share of the memory
// free at the stream's first traceback.
constexpr int64_t kTbCapMax = (int64_t)16 << 30, kTbCapMin = (int64_t)1 << 30;
constexpr double kTbFreeShare = 0.3;

// Tries sizes from `want` down to `least`, each half the one before, until
// alloc(bytes) takes one.  Returns it (0: none).
template <class Alloc>
size_t alloc_between(size_t want, size_t least, Alloc &&alloc)
{
    for (size_t bytes = want;; bytes = std::max(bytes / 2, least)) {
        if (alloc(bytes)) return bytes;
        if (bytes <= least) return 0;
    }
}

}  // namespace swgb
