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

// Scratch of a plan, which knows its classes: boundary rows for every warp of the
// score launches that need them, and the traceback's for the worst case of the
// shape.  Every window may lie inside the band, so a chunk window is at most the
// class's longest window; the slots are for the warps that the classes' pairs can
// keep busy (64 pairs of 100 x 150: 2 MB, where every warp of every launch took
// 1.8 GB; 16,384 of 100 x 200: 0.25 GB and 2.3).
inline void plan_budgets(const ClassInfo &ci, const PlanParams &pp, bool cigar, int64_t &bnd_bytes, int64_t &tb_bytes)
{
    int64_t slot_s[N_SCORE_VARIANTS] = {};
    for (int c = 0; c < N_CLASS; ++c) {
        if (!ci.count[c]) continue;
        const int mode = c / N_MCLASS;
        const int32_t mm = ci.max_m[c], mn = ci.max_n[c];
        int lanes = 1, ri = 0;
        score_plan_of(mode, mm, (int64_t)pp.sc.ma * std::min(mm, mn), pp.ov, pp.n_overrides, lanes, ri);
        const int rows = score_rows_at(ri);
        if ((mm + lanes * rows - 1) / (lanes * rows) > 1) {
            const int v = ri * N_VMODES + score_vmode(mode, (int64_t)pp.sc.ma * std::min(mm, mn), pp.sc, true);
            slot_s[v] = std::max<int64_t>(slot_s[v], (int64_t)(32 / lanes) * 16 * mn);
        }
    }
    int nb = 0;
    int64_t per = 0;
    for (int v = 0; v < N_SCORE_VARIANTS; ++v)
        if (slot_s[v]) {
            ++nb;
            per = std::max(per, slot_s[v] * pp.score_warps[v]);
        }
    bnd_bytes = std::max<int64_t>(nb * ((per + 255) & ~(int64_t)255), 256);
    tb_bytes = 0;
    if (!cigar) return;
    // the row checkpoints of every class, and per 16-bit launch a slot, the widest
    // of the classes it may serve, for every warp that they may give a task
    int64_t all = 0, ck = 0;
    for (int c = N_MCLASS; c < N_CLASS; ++c) all += ci.count[c];
    int64_t slot_v[N_TB_VARIANTS] = {}, tasks_v[N_TB_VARIANTS] = {};
    for (int c = 0; c < N_CLASS; ++c) {
        if (!ci.count[c]) continue;
        const int mode = c / N_MCLASS;
        const int32_t mm = ci.max_m[c], mn = std::max(ci.max_n[c], 1);
        const int64_t cnt = ci.count[c], chunks = (mm + TB_ROWS - 1) / TB_ROWS;
        auto add = [&](int64_t w, int part, int lanes) {
            TbPartPlan t{};
            const int64_t slot =
                tb_part_shape(mode, pp.allow16 != 0, 64, mm, chunks * w, (int32_t)w, part, pp.sc, lanes, t);
            const int v = tb_launch_first(t.variant);
            slot_v[v] = std::max(slot_v[v], (slot + 63) & ~(int64_t)63);
            // (a part's last task may be short)
            tasks_v[v] += v < N_TB16_VARIANTS ? (cnt * lanes + 63) / 64 + 1 : cnt;
        };
        if (pp.allow16 && mode != MODE_I32) {
            ck += 16 * std::max(ck_class_units(cnt, (int64_t)ci.sum_n[c], mm, mn, 1, 50),
                                ck_class_units(cnt, (int64_t)ci.sum_n[c], mm, mn, 32, 50));
            // every part at its widest window, and every number of lanes that
            // it may get: fewer pairs in a part only ask for more
            const int32_t widest[kTbParts] = {mn, kTbWide, kTbMid};
            for (int part = 0; part < kTbParts; ++part) {
                if ((part == 0 && mn <= kTbWide) || (part == 1 && mn <= kTbMid)) continue;
                for (int lanes = tb_part_lanes(false, part, all, all, cnt, mm, pp.tb_warps[0]); lanes <= 16; lanes *= 2)
                    add(std::min(mn, widest[part]), part, lanes);
            }
        } else {
            // the widest window, and the widest one-lane tile
            add(mn, 0, 1);
            add(std::max<int64_t>(1, std::min<int64_t>(mn, kTiledLaneWords / chunks)), 0, 1);
        }
    }
    const int64_t cap = kTbCapMax / 4;  // words
    int64_t all16 = 0;  // the 16-bit launches run at once
    for (int v = 0; v < N_TB_VARIANTS; ++v) {
        const int64_t warps = std::min<int64_t>(pp.tb_warps[v], tasks_v[v]);
        const int64_t words = std::max(std::min(warps * slot_v[v], cap), std::min<int64_t>(warps, 4) * slot_v[v]);
        if (v < N_TB16_VARIANTS) all16 += words;
        else tb_bytes = std::max(tb_bytes, 4 * words);
    }
    tb_bytes = std::max(tb_bytes, 4 * std::min(all16, 2 * cap));
    tb_bytes += 1 << 20;  // (roundings)
    // the planner lets checkpoints take three quarters of the scratch
    tb_bytes = std::max(tb_bytes + std::min(ck, kTbCapMax), (std::min(ck, kTbCapMax) + 2) / 3 * 4);
}

}  // namespace swgb
