// sw_classify.cuh -- a pair's length class, as the classification kernels
// compute it.
#pragma once
#include "sw_device.cuh"
#include "swgb_internal.h"

namespace swgb {

// One pair's sort key (class and window bucket), -1 when nothing is to be
// aligned: its outputs are then written here (or the status for an invalid
// pair).  m, n: its lengths.
__device__ __forceinline__ int32_t classify_pair(const PairSet &ps, int64_t n_reads, int64_t p, const Scoring &sc,
                                                 int score_setting, int32_t *status, int32_t *out_score,
                                                 int32_t *out_end, int32_t *cig_n, int32_t &cls, int64_t &m,
                                                 int64_t &n)
{
    const int64_t rd = ps.pair_read ? ps.pair_read[p] : p;
    bool bad = rd < 0 || rd >= n_reads;
    if (!bad) {
        const int64_t r0 = ps.read_off[rd], r1 = ps.read_off[rd + 1];
        const int64_t w0 = ps.win_off[p], w1 = ps.win_off[p + 1];
        m = r1 - r0;
        n = w1 - w0;
        bad = r0 < 0 || w0 < 0 || m < 1 || m > SW_MAX_READ_LEN || n < 0 || n > SW_MAX_WINDOW_LEN;
    }
    if (bad) {
        atomicOr(status, ST_BAD_INPUT);
        return -1;
    }
    const bool masked = ps.mask && !ps.mask[p];
    if (masked || n == 0) {
        // not selected: no alignment; an empty window aligns nothing: score
        // 0, no end cell, no CIGAR
        out_score[p] = masked ? -1 : 0;
        out_end[2 * p] = -1;
        out_end[2 * p + 1] = -1;
        if (cig_n) cig_n[p] = 0;
        return -1;
    }
    const int64_t hmax = (int64_t)sc.ma * (m < n ? m : n);
    cls = score_mode_for(hmax, score_setting) * N_MCLASS + mclass_of((int32_t)m);
    int nb = (int)((n - 1) >> 5);
    nb = nb > N_NBUCKET - 1 ? N_NBUCKET - 1 : nb;
    return cls * N_NBUCKET + (N_NBUCKET - 1 - nb);
}

}  // namespace swgb
