// sw_devplan.cu -- launch planning on the device.
//
// The paper hands whole batches to OpenMP threads and balances the thread
// counts of its stages by hand (Section 3.4, Section 4.3).  Here a batch is
// sorted into length classes on the GPU, and two one-block kernels plan the
// launches from the classification's per-class facts, so that the host
// enqueues a fixed sequence of launches and never waits for the device:
//
//   k_plan_score  per class the lanes per pair and rows per lane (the cost
//                 model of score_plan_of), the class's place in the sorted
//                 order, its score variant (compiled rows x arithmetic
//                 mode), the chunk-boundary scratch of classes whose
//                 reads need several row chunks, and which classes keep row
//                 checkpoints for the traceback;
//   k_plan_tb     per class and part (pairs with wide windows, the rest) the
//                 traceback kernel, its lanes per pair and slab sizes
//                 (tb_part_shape), and per traceback variant the size of a
//                 warp's scratch slot and how many warps fit the budget.
//
// Each variant's list is ordered longest reads first, so the persistent
// launches end on short work.
#include "sw_device.cuh"
#include "swgb_internal.h"

namespace swgb {

__global__ void __launch_bounds__(kPlanThreads) k_plan_score(const ClassInfo *__restrict__ info, const PlanParams pp,
                                                             DevScorePlan *__restrict__ out,
                                                             int32_t *__restrict__ status)
{
    __shared__ int32_t s_var[N_CLASS], s_cnt[N_CLASS], s_bnd[N_CLASS], s_lanes[N_CLASS], s_ck[N_CLASS];
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        const int32_t cnt = info->count[c];
        int32_t var = -1, bnd = 0, lanes = 1, ck = 0;
        if (cnt > 0) {
            const int mode = c / N_MCLASS;
            const int32_t mm = info->max_m[c], mn = info->max_n[c];
            int ri = 0;
            const int64_t hmax = (int64_t)pp.sc.ma * min(mm, mn);
            score_plan_of(mode, mm, hmax, pp.ov, pp.n_overrides, lanes, ri);
            const int vmode = score_vmode(mode, hmax, pp.sc);
            // a class with fewer tasks than half its launch's warps (a small
            // batch) finishes when one task does: fewer rows per lane, on
            // more lanes, shorten the task while it still fits one row chunk
            // (not when an override chose the plan)
            bool chosen = false;
            for (int i = 0; i < pp.n_overrides; ++i) chosen |= mm <= pp.ov[i].max_read_len;
            while (!chosen && ri > 0) {
                const int64_t per_warp = (int64_t)(32 / lanes) * (mode != MODE_I32 ? 2 : 1);
                const int64_t tasks = (cnt + per_warp - 1) / per_warp;
                if (2 * tasks >= pp.score_warps[ri * N_VMODES + vmode]) break;
                const int t2 = (mm + score_rows_at(ri - 1) - 1) / score_rows_at(ri - 1);
                if (t2 > 32) break;
                --ri;
                lanes = t2;
            }
            const int rows = score_rows_at(ri);
            const int chunks = (mm + lanes * rows - 1) / (lanes * rows);
            // per group: two buffers x longest window x (H, F) x 4 bytes
            bnd = chunks > 1 ? 16 * mn : 0;
            var = ri * N_VMODES + vmode;
            if (pp.ck_bytes > 0 && mode != MODE_I32) ck = ck_block_rows(rows);
        }
        s_var[c] = var;
        s_cnt[c] = cnt;
        s_bnd[c] = bnd;
        s_lanes[c] = lanes;
        s_ck[c] = ck;
        out->cls_count[c] = cnt;
        out->cls_lanes[c] = lanes;
        out->cls_bnd_bytes[c] = bnd;
    }
    __syncthreads();
    // the first warp finishes: class starts (a warp scan over the counts),
    // then each variant's class list, longest reads first (classes are
    // mode-major, so within a variant -- one mode -- a larger class index is
    // a longer read class), built with ballots
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
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
            if (c < N_CLASS) {
                out->cls_start[c] = run;
                run += s_cnt[c];
            }
        }
    }
    // checkpoints: blocks are doubled until the most they may take fits the
    // pool (a block of the whole read needs none)
    {
        const int64_t limit = min(pp.ck_bytes / 16, (int64_t)0xFFFFFFF0u);
        int64_t used = 0;
        int shift = 0;
        for (;; ++shift) {
            used = 0;
            for (int c = lane; c < N_CLASS; c += 32)
                if (s_ck[c])
                    used += ck_class_units(s_cnt[c], (int64_t)info->sum_n[c], info->max_m[c], info->max_n[c],
                                           s_lanes[c], s_ck[c] << shift);
            for (int d = 16; d; d >>= 1) used += __shfl_xor_sync(0xffffffffu, used, d);
            if (used <= limit) break;  // at the latest when no read is longer than its block
        }
        for (int c = lane; c < N_CLASS; c += 32) out->cls_ck[c] = s_ck[c] << shift;
        if (lane == 0) out->ck_units = (used + 15) & ~(int64_t)15;  // 256-byte alignment
    }
    int nb = 0;
    int32_t n_v[N_SCORE_VARIANTS];
    int64_t slot_v[N_SCORE_VARIANTS];
    for (int v = 0; v < N_SCORE_VARIANTS; ++v) {
        int32_t n = 0;
        int64_t slot = 0;
        for (int c0 = N_CLASS - 1; c0 >= 0; c0 -= 32) {
            const int c = c0 - lane;
            const bool hit = c >= 0 && s_var[c] == v;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (hit) {
                out->var_cls[v][n + __popc(m & lt)] = (int16_t)c;
                slot = max(slot, (int64_t)(32 / s_lanes[c]) * s_bnd[c]);  // a warp's groups
            }
            n += __popc(m);
        }
        for (int d = 16; d; d >>= 1) slot = max(slot, __shfl_xor_sync(0xffffffffu, slot, d));
        n_v[v] = n;
        slot_v[v] = slot;
        nb += slot > 0;
    }
    if (lane != 0) return;
    const int64_t share = nb ? (pp.score_bnd_bytes / nb) & ~(int64_t)255 : 0;
    int64_t off = 0;
    for (int v = 0; v < N_SCORE_VARIANTS; ++v) {
        out->var_n[v] = n_v[v];
        out->var_bnd_warps[v] = 0;
        out->var_bnd_offset[v] = 0;
        out->var_bnd_slot[v] = slot_v[v];
        if (slot_v[v] > 0) {
            const int64_t w = min((int64_t)pp.score_warps[v], share / slot_v[v]);
            if (w < 1) atomicOr(status, ST_UNSUPPORTED);  // one warp's rows do not fit the scratch
            out->var_bnd_warps[v] = (int32_t)w;
            out->var_bnd_offset[v] = off;
            off += share;
        }
    }
}

__global__ void __launch_bounds__(kPlanThreads) k_plan_tb(const ClassInfo *__restrict__ info,
                                                          const TbClassInfo *__restrict__ ti,
                                                          const DevScorePlan *__restrict__ sp, const PlanParams pp,
                                                          DevTbPlan *__restrict__ out, int32_t *__restrict__ status)
{
    __shared__ int64_t s_slot[N_TB_PARTS];
    __shared__ int8_t s_pv[N_TB_PARTS];  // each part's variant (-1: none)
    __shared__ int32_t s_n16;            // pairs of the 16-bit classes
    if (threadIdx.x == 0) s_n16 = 0;
    __syncthreads();
    if (threadIdx.x < N_CLASS && threadIdx.x >= N_MCLASS && info->count[threadIdx.x] > 0)
        atomicAdd(&s_n16, info->count[threadIdx.x]);
    __syncthreads();
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        const int32_t cnt = info->count[c];
        const int32_t big = ti->n_big[c];
        const int32_t counts[2] = {big, cnt - big};
        const int32_t starts[2] = {sp->cls_start[c], sp->cls_start[c] + big};
        for (int part = 0; part < 2; ++part) {
            TbPartPlan t{};
            t.cls = c;
            t.part = part;
            t.start = starts[part];
            t.count = counts[part];
            t.variant = -1;
            int64_t slot = 0;
            if (t.count > 0) {
                const int64_t need = ti->max_need[c] > 1 ? ti->max_need[c] : 1;
                // a batch too small to give a task (64 / T pairs) to a
                // quarter of the warps of a launch spreads each two pairs
                // over more lanes, and so does a small part of long reads
                // (its tasks are many blocks one after another): the tasks
                // then finish sooner, which is what the call waits for
                int lanes = part == 0 ? 8 : 1;  // wide windows: see kTbWide
                const int64_t enough = (int64_t)pp.tb_warps[0] * 16;
                while (lanes < 8 && ((int64_t)s_n16 * lanes < enough ||
                                     (info->max_m[c] > 512 && (int64_t)t.count * lanes < enough)))
                    lanes *= 2;
                slot = tb_part_shape(c / N_MCLASS, pp.allow16 != 0, sp->cls_ck[c], info->max_m[c], need,
                                     ti->max_wcap[part][c], part, pp.sc, lanes, t);
            }
            out->part[2 * c + part] = t;
            s_slot[2 * c + part] = slot;
            s_pv[2 * c + part] = (int8_t)t.variant;
        }
    }
    __syncthreads();
    // the first warp finishes: each variant's part list (longest reads
    // first, wide part first), its slot size, and the split
    if (threadIdx.x >= 32) return;
    const int lane = threadIdx.x;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t ck_words = 4 * sp->ck_units;
    const int64_t total = pp.tb_bytes / 4 - ck_words;
    int64_t split16 = 0, split32 = 0;
    for (int v = 0; v < N_TB_VARIANTS; ++v) {
        int32_t n = 0;
        int64_t slot = 0;
        for (int q0 = N_TB_PARTS - 1; q0 >= 0; q0 -= 32) {
            // parts 2c (wide) and 2c + 1 of class c, classes descending
            const int qi = q0 - lane;
            const int q = qi >= 0 ? (qi ^ 1) : -1;
            const bool hit = q >= 0 && s_pv[q] == v;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (hit) {
                out->var_part[v][n + __popc(m & lt)] = (int16_t)q;
                slot = max(slot, s_slot[q]);
                (v < N_TB16_VARIANTS ? split16 : split32) += out->part[q].count;
            }
            n += __popc(m);
        }
        for (int d = 16; d; d >>= 1) slot = max(slot, __shfl_xor_sync(0xffffffffu, slot, d));
        if (lane == 0) {
            // a slot per warp, as many warps as fit (the launches run one
            // after another, each with everything the checkpoints leave)
            const int64_t words = (slot + 63) & ~(int64_t)63;  // 256-byte alignment
            const int64_t w = n ? min((int64_t)pp.tb_warps[v], total / max(words, (int64_t)1)) : 0;
            if (n && w < 1) atomicOr(status, ST_UNSUPPORTED);  // one warp's slot does not fit the scratch
            out->var_n[v] = n;
            out->var_slot_words[v] = words;
            out->var_slot_offset[v] = ck_words;
            out->var_warps[v] = (int32_t)w;
        }
    }
    for (int d = 16; d; d >>= 1) {
        split16 += __shfl_xor_sync(0xffffffffu, split16, d);
        split32 += __shfl_xor_sync(0xffffffffu, split32, d);
    }
    if (lane == 0) {
        out->split[0] = split16;
        out->split[1] = split32;
    }
}

int launch_plan_score(const ClassInfo *info, const PlanParams &pp, DevScorePlan *out, int32_t *status,
                      cudaStream_t st)
{
    k_plan_score<<<1, kPlanThreads, 0, st>>>(info, pp, out, status);
    count_launch();
    return launch_status();
}

int launch_plan_tb(const ClassInfo *info, const TbClassInfo *ti, const DevScorePlan *sp, const PlanParams &pp,
                   DevTbPlan *out, int32_t *status, cudaStream_t st)
{
    k_plan_tb<<<1, kPlanThreads, 0, st>>>(info, ti, sp, pp, out, status);
    count_launch();
    return launch_status();
}

}  // namespace swgb
