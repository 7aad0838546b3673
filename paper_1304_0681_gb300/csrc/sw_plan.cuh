// sw_plan.cuh -- launch planning on the device (bodies of the planner kernels).
//
// The paper hands whole batches to OpenMP threads and balances the thread
// counts of its stages by hand (Section 3.4, Section 4.3).  Here a batch is
// sorted into length classes on the GPU, and one block each plans the
// launches from the classification's per-class facts, so that the host
// enqueues a fixed sequence of launches and never waits for the device:
//
//   plan_score    per class the lanes per pair and rows per lane (the cost
//                 model of score_plan_of), the class's place in the sorted
//                 order, its score variant (compiled rows x arithmetic
//                 mode), the chunk-boundary scratch of classes whose
//                 reads need several row chunks, and which classes keep row
//                 checkpoints for the traceback;
//   plan_tb       per class and part (pairs with wide windows, the rest) the
//                 traceback kernel, its lanes per pair and slab sizes
//                 (tb_part_shape), and per traceback variant the size of a
//                 warp's scratch slot and how many warps fit the budget.
//
// Each variant's list is ordered longest reads first, so the persistent
// launches end on short work.
//
// A batch has few classes: the first warp lists them once, and every later
// step runs over that list, a lane per launch variant.
#pragma once
#include "sw_device.cuh"
#include "swgb_internal.h"

namespace swgb {

// The non-empty classes (count[c] > 0), largest index first, by the first
// warp; returns how many.
__device__ __forceinline__ int list_classes(const int32_t *count, int16_t *list)
{
    const int lane = threadIdx.x & 31;
    int n = 0;
    for (int c0 = N_CLASS - 1; c0 >= 0; c0 -= 32) {
        const int c = c0 - lane;
        const bool hit = c >= 0 && count[c] > 0;
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (hit) list[n + __popc(m & ((1u << lane) - 1u))] = (int16_t)c;
        n += __popc(m);
    }
    __syncwarp();
    return n;
}

// The score plan of a class in a batch that fills the GPU: lanes per group,
// rows index and kernel mode.  Returns whether an override gives it.
__device__ __forceinline__ bool plan_class(const PlanParams &pp, int mode, int32_t mm, int32_t mn, int &lanes, int &ri,
                                           int &vmode)
{
    const int64_t hmax = (int64_t)pp.sc.ma * min(mm, mn);
    score_plan_of(mode, mm, hmax, pp.ov, pp.n_overrides, lanes, ri);
    vmode = score_vmode(mode, hmax, pp.sc, mm > lanes * score_rows_at(ri));
    for (int i = 0; i < pp.n_overrides; ++i)
        if (mm <= pp.ov[i].max_read_len) return true;
    if (pp.small && !small_body(ri, vmode)) {
        // not in a small batch's one launch: the next larger row count (its
        // lanes then cover the read in no more chunks)
        ++ri;
        lanes = min(32, (mm + score_rows_at(ri) - 1) / score_rows_at(ri));
    }
    return false;
}

// Issue slots of a class's task (a warp's groups) at a rows index, in the
// units of score_plan_of's cost.
__device__ __forceinline__ int64_t task_slots(int mode, int ri, int lanes, int32_t mean_n)
{
    return (int64_t)((mode != MODE_I32 ? mean_n / 2 : mean_n) + lanes) * (13 * score_rows_at(ri) + 80);
}

// Tasks of cnt pairs at this many lanes per group.
__device__ __forceinline__ uint32_t class_tasks(int mode, int32_t cnt, int lanes)
{
    const uint32_t per_warp = (uint32_t)(32 / lanes) * (mode != MODE_I32 ? 2u : 1u);
    return ((uint32_t)cnt + per_warp - 1u) / per_warp;
}

// Fewer rows per lane, on more lanes, make a class's tasks shorter and more,
// and cost slots.
//
// A class that is most of its batch takes the plan with the least estimated
// time, of those with the read in one row chunk.  A launch's warps take tasks
// in waves; a warp by itself issues an instruction every 2.7 cycles, a scheduler
// with enough warps one every 1.25, so a wave takes a task's slots times the
// warps on a scheduler or times 13/6, whichever is more.  Score pass with its
// launches at 16,384 pairs of 100 x 200: 50 rows 0.209 ms, 32 0.203, 25 0.175
// (taken), 20 0.154, 16 0.165, 8 0.183; of 150 x 250: 50 rows 0.256, 25 0.209
// (taken), 16 0.244; 40,000 of 250 x 350: 50 rows 0.907, 25 0.863 (taken), 16
// 0.948.  From about 100,000 pairs on it is the full GPU's plan.
//
// The other classes run beside more work than their own, and so do a small
// batch's, whose launch holds every plan: fewer rows while a class has fewer
// tasks than half its launch's warps (20,000 reads of six lengths: the estimate
// above took 2.8 ms, this 1.5).
__device__ __forceinline__ void plan_rows(const PlanParams &pp, int mode, int vmode, int32_t cnt, int32_t mm,
                                          int32_t mean_n, bool most, int &lanes, int &ri)
{
    if (pp.small || !most) {
        while (ri > 0) {
            if (2 * (int64_t)class_tasks(mode, cnt, lanes) >= pp.score_warps[ri * N_VMODES + vmode]) break;
            const int r2 = pp.small && !small_rows(ri - 1) ? ri - 2 : ri - 1;
            const int t2 = (mm + score_rows_at(r2) - 1) / score_rows_at(r2);
            if (t2 > 32) break;
            ri = r2;
            lanes = t2;
        }
        return;
    }
    int64_t best = -1;
    for (int r = ri; r >= 0; --r) {
        const int t = (mm + score_rows_at(r) - 1) / score_rows_at(r);
        if (t > 32) break;
        const uint32_t tasks = class_tasks(mode, cnt, t), warps = (uint32_t)pp.score_warps[r * N_VMODES + vmode];
        // in sixths of a task's slots
        const uint32_t sch = (uint32_t)pp.schedulers;
        auto wave = [&](uint32_t w) { return max(13u, 6u * ((w + sch - 1u) / sch)); };
        const uint32_t full = tasks / warps, last = tasks - full * warps;
        const int64_t cost =
            task_slots(mode, r, t, mean_n) * ((int64_t)full * wave(warps) + (last ? wave(last) : 0u));
        if (best < 0 || cost < best) {
            best = cost;
            ri = r;
            lanes = t;
        }
    }
}

// Whole block; the first warp finishes (no barrier at the end).
__device__ __forceinline__ void plan_score(const ClassInfo *info, const PlanParams &pp, DevScorePlan *out,
                                           int32_t *status)
{
    __shared__ int32_t s_var[N_CLASS], s_cnt[N_CLASS], s_bnd[N_CLASS], s_lanes[N_CLASS], s_ck[N_CLASS];
    __shared__ int16_t s_list[N_CLASS];
    __shared__ int32_t s_pipe_tasks;
    __shared__ unsigned long long s_pipe_bytes, s_slots, s_work[N_CLASS];
    if (threadIdx.x == 0) {
        s_pipe_tasks = 0;
        s_pipe_bytes = 0;
        s_slots = 0;
    }
    __syncthreads();
    auto long_class = [&](int c) { return pp.small && block_task_class(c, info->max_m[c]); };
    auto mean_n = [&](int c) { return (int32_t)__fdividef((float)info->sum_n[c], (float)info->count[c]); };
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        const int32_t cnt = info->count[c];
        if (cnt == 0) continue;
        if (long_class(c)) atomicAdd(&s_pipe_tasks, (int32_t)block_task_tasks(cnt));
        const int mode = c / N_MCLASS;
        int lanes = 1, ri = 0, vmode = 0;
        const bool fixed = plan_class(pp, mode, info->max_m[c], info->max_n[c], lanes, ri, vmode);
        const unsigned long long work =
            (unsigned long long)class_tasks(mode, cnt, lanes) * (unsigned long long)task_slots(mode, ri, lanes, mean_n(c));
        s_var[c] = fixed ? ~(ri * N_VMODES + vmode) : ri * N_VMODES + vmode;
        s_lanes[c] = lanes;
        s_work[c] = work;
        atomicAdd(&s_slots, work);
    }
    __syncthreads();
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        const int32_t cnt = info->count[c];
        int32_t var = -1, bnd = 0, ck = 0;
        int lanes = 1;
        if (cnt > 0) {
            const int mode = c / N_MCLASS;
            const int32_t mm = info->max_m[c], mn = info->max_n[c];
            int ri = 0, vmode = mode;
            int64_t pipe = -1;
            if (long_class(c) && s_pipe_tasks <= pp.score_warps[0] / kPipeWarps) {
                const unsigned long long need = (unsigned long long)block_task_need(cnt, mn);
                const unsigned long long at = atomicAdd(&s_pipe_bytes, need);
                if (at + need <= (unsigned long long)pp.pipe_bytes) pipe = (int64_t)at;
            }
            out->cls_pipe[c] = pipe;
            if (pipe >= 0) {
                lanes = 32;
                ri = pipe_rows_idx(mm);
                vmode = MODE_I16W;
            } else {
                const bool fixed = s_var[c] < 0, most = 4 * s_work[c] >= 3 * s_slots;
                const int v = fixed ? ~s_var[c] : s_var[c];
                ri = v / N_VMODES;
                vmode = v % N_VMODES;
                lanes = s_lanes[c];
                if (!fixed) plan_rows(pp, mode, vmode, cnt, mm, mean_n(c), most, lanes, ri);
            }
            const int rows = score_rows_at(ri);
            const int chunks = (mm + lanes * rows - 1) / (lanes * rows);
            // per group: two buffers x longest window x (H, F) x 4 bytes
            bnd = chunks > 1 && pipe < 0 ? 16 * mn : 0;
            var = ri * N_VMODES + vmode;
            if (pp.ck_bytes > 0 && mode != MODE_I32) ck = ck_block_rows(rows);
            out->cls_count[c] = cnt;
            out->cls_lanes[c] = lanes;
            out->cls_bnd_bytes[c] = pipe >= 0 ? 16 * mn : bnd;
        }
        s_var[c] = var;
        s_cnt[c] = cnt;
        s_bnd[c] = bnd;
        s_lanes[c] = lanes;
        s_ck[c] = ck;
    }
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    // class starts in the sorted order: a warp scan over the counts
    {
        constexpr int PER = (N_CLASS + 31) / 32;
        int32_t sum = 0;
        for (int i = 0; i < PER; ++i) {
            const int c = lane * PER + i;
            if (c < N_CLASS) sum += s_cnt[c];
        }
        int32_t x = sum;
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        int32_t run = x - sum;
        for (int i = 0; i < PER; ++i) {
            const int c = lane * PER + i;
            if (c < N_CLASS && s_cnt[c]) {
                out->cls_start[c] = run;
                run += s_cnt[c];
            }
        }
    }
    const int n_list = list_classes(s_cnt, s_list);
    // checkpoints: blocks are doubled until the most they may take fits the
    // pool (a block of the whole read needs none)
    {
        const int64_t limit = min(pp.ck_bytes / 16, (int64_t)0xFFFFFFF0u);
        int64_t used = 0;
        int shift = 0;
        for (;; ++shift) {
            used = 0;
            for (int q = lane; q < n_list; q += 32) {
                const int c = s_list[q];
                if (s_ck[c])
                    used += ck_class_units(s_cnt[c], (int64_t)info->sum_n[c], info->max_m[c], info->max_n[c],
                                           s_lanes[c], s_ck[c] << shift);
            }
            for (int d = 16; d; d >>= 1) used += __shfl_xor_sync(0xffffffffu, used, d);
            if (used <= limit) break;  // at the latest when no read is longer than its block
        }
        for (int q = lane; q < n_list; q += 32) out->cls_ck[s_list[q]] = s_ck[s_list[q]] << shift;
        if (lane == 0) out->ck_units = (used + 15) & ~(int64_t)15;  // 256-byte alignment
    }
    // each variant's class list, longest reads first (classes are mode-major,
    // so within a variant -- one mode -- a larger class index is a longer
    // read class)
    static_assert(N_SCORE_VARIANTS <= 32, "a lane per variant");
    int32_t n = 0;
    int64_t slot = 0;
    for (int q = 0; q < n_list; ++q) {
        const int c = s_list[q];
        if (s_var[c] == lane) {
            out->var_cls[lane][n++] = (int16_t)c;
            slot = max(slot, (int64_t)(32 / s_lanes[c]) * s_bnd[c]);  // a warp's groups
        }
    }
    const unsigned chunked = __ballot_sync(0xffffffffu, slot > 0);
    if (lane < N_SCORE_VARIANTS) {
        const int nb = __popc(chunked);
        const int64_t share = nb ? (pp.score_bnd_bytes / nb) & ~(int64_t)255 : 0;
        int64_t w = 0;
        if (slot > 0) {
            w = min((int64_t)pp.score_warps[lane], share / slot);
            if (w < 1) atomicOr(status, ST_UNSUPPORTED);  // one warp's rows do not fit the scratch
        }
        out->var_n[lane] = n;
        out->var_bnd_warps[lane] = (int32_t)w;
        out->var_bnd_offset[lane] = __popc(chunked & ((1u << lane) - 1u)) * share;
        out->var_bnd_slot[lane] = slot;
    }
}

// Whole block.  The 16-bit launches run at once (a few wide pairs' tasks are
// long and leave the SMs half empty), each with its part of the scratch: a
// slot for every warp that gets a task while they fit, else a slot each and
// the rest in proportion.  Where not even one slot each fits, every 16-bit
// part takes the 16-lane launch, whose slots are the smallest.  The int32
// launches follow, each with all of the scratch.
__device__ __forceinline__ void plan_tb(const ClassInfo *info, const TbClassInfo *ti, const DevScorePlan *sp,
                                        const PlanParams &pp, DevTbPlan *out, int32_t *status)
{
    __shared__ int64_t s_slot[N_TB_PARTS];
    __shared__ int32_t s_tbcnt[N_CLASS], s_part[N_TB_PARTS];
    __shared__ int8_t s_pv[N_TB_PARTS];  // each part's variant (-1: none)
    __shared__ int16_t s_tblist[N_CLASS];
    __shared__ int32_t s_n16[kTbParts];  // pairs of the 16-bit classes by part
    __shared__ int32_t s_retry;
    if (threadIdx.x < kTbParts) s_n16[threadIdx.x] = 0;
    __syncthreads();
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        const int32_t cnt = s_tbcnt[c] = info->count[c];
        if (c >= N_MCLASS && cnt > 0) {
            atomicAdd(&s_n16[0], ti->n_part[0][c]);
            atomicAdd(&s_n16[1], ti->n_part[1][c]);
            atomicAdd(&s_n16[2], cnt);
        }
    }
    __syncthreads();
    for (bool one_launch = pp.small != 0;; one_launch = true) {
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        const int32_t cnt = s_tbcnt[c];
        if (!cnt) continue;
        const int32_t n0 = ti->n_part[0][c], n1 = ti->n_part[1][c];
        const int32_t counts[kTbParts] = {n0, n1, cnt - n0 - n1};
        int32_t start = sp->cls_start[c];
        for (int part = 0; part < kTbParts; ++part) {
            TbPartPlan t{};
            t.cls = c;
            t.part = part;
            t.start = start;
            t.count = counts[part];
            t.variant = -1;
            start += t.count;
            int64_t slot = 0;
            if (t.count > 0) {
                const int64_t need = ti->max_need[c] > 1 ? ti->max_need[c] : 1;
                const int64_t all = s_n16[2];
                const int lanes = tb_part_lanes(one_launch, part, all, part < 2 ? s_n16[part] : all, cnt, info->max_m[c],
                                                pp.tb_warps[0]);
                slot = tb_part_shape(c / N_MCLASS, pp.allow16 != 0, sp->cls_ck[c], info->max_m[c], need,
                                     ti->max_wcap[part][c], part, pp.sc, lanes, t);
                out->part[kTbParts * c + part] = t;
            }
            s_slot[kTbParts * c + part] = slot;
            s_part[kTbParts * c + part] = t.count;
            s_pv[kTbParts * c + part] = (int8_t)t.variant;
        }
    }
    __syncthreads();
    // the first warp finishes: each variant's part list (longest reads
    // first, wide part first), its slots, and the split
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const int n_list = list_classes(s_tbcnt, s_tblist);
        const int64_t ck_words = 4 * sp->ck_units;
        const int64_t total = pp.tb_bytes / 4 - ck_words;
        const int32_t per_task = lane < N_TB16_VARIANTS ? 64 / tb16_variant_lanes(lane) : 1;
        int32_t n = 0;
        int64_t words = 0, pairs = 0, tasks = 0;
        for (int q = 0; q < n_list; ++q)
            for (int part = 0; part < kTbParts; ++part) {
                const int x = kTbParts * s_tblist[q] + part;
                if (s_pv[x] == lane) {
                    out->var_part[lane][n++] = (int16_t)x;
                    words = max(words, s_slot[x]);
                    pairs += s_part[x];
                    tasks += (s_part[x] + per_task - 1) / per_task;
                }
            }
        // the variants of one launch share its slots
        {
            const int64_t w = __shfl_xor_sync(0xffffffffu, words, 1), t = __shfl_xor_sync(0xffffffffu, tasks, 1);
            if (lane < 4) {
                words = max(words, w);
                tasks += t;
            }
        }
        words = (words + 63) & ~(int64_t)63;  // 256-byte alignment
        const int64_t warps = lane < N_TB_VARIANTS ? min((int64_t)pp.tb_warps[lane], tasks) : 0;
        const bool leads = lane < N_TB16_VARIANTS && (lane >= 4 || !(lane & 1)) && warps > 0;
        const int64_t one = leads ? words : 0, more = leads ? (warps - 1) * words : 0;
        int64_t ones = one, mores = more;
        for (int d = 16; d; d >>= 1) {
            ones += __shfl_xor_sync(0xffffffffu, ones, d);
            mores += __shfl_xor_sync(0xffffffffu, mores, d);
        }
        int64_t w = leads ? 1 : 0;
        if (leads) {
            if (ones + mores <= total) w = warps;
            else if (ones < total) w += (int64_t)((double)(total - ones) * ((double)more / (double)mores)) / words;
        }
        const int64_t area = w * words;
        int64_t at = area;
        for (int d = 1; d < 32; d <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, at, d);
            if (lane >= d) at += y;
        }
        at -= area;
        {
            const int64_t w0 = __shfl_sync(0xffffffffu, w, lane & ~1), at0 = __shfl_sync(0xffffffffu, at, lane & ~1);
            if (lane < 4) {
                w = w0;
                at = at0;
            }
        }
        if (lane >= N_TB16_VARIANTS && lane < N_TB_VARIANTS) {
            // int32: as many warps as fit all of the scratch (the checkpoints
            // have been read by then)
            w = n ? min((int64_t)pp.tb_warps[lane], pp.tb_bytes / 4 / max(words, (int64_t)1)) : 0;
            at = -ck_words;
            if (n && w < 1) atomicOr(status, ST_UNSUPPORTED);  // one warp's slot does not fit the scratch
        }
        if (lane == 0) {
            s_retry = ones > total && !one_launch;
            if (ones > total && one_launch) atomicOr(status, ST_UNSUPPORTED);
        }
        int64_t split16 = lane < N_TB16_VARIANTS ? pairs : 0, split32 = lane >= N_TB16_VARIANTS ? pairs : 0;
        for (int d = 16; d; d >>= 1) {
            split16 += __shfl_xor_sync(0xffffffffu, split16, d);
            split32 += __shfl_xor_sync(0xffffffffu, split32, d);
        }
        if (lane < N_TB_VARIANTS) {
            out->var_n[lane] = n;
            out->var_slot_words[lane] = words;
            out->var_slot_offset[lane] = ck_words + at;
            out->var_warps[lane] = (int32_t)w;
        }
        if (lane == 0) {
            out->split[0] = split16;
            out->split[1] = split32;
        }
    }
    __syncthreads();
    if (!s_retry) break;
    __syncthreads();
    }
}

}  // namespace swgb
