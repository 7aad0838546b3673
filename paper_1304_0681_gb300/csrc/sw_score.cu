// sw_score.cu -- launches of the score pass, and its kernels without
// checkpoints (sw_score_kernel.cuh).
#include <algorithm>

#include "sw_score_kernel.cuh"

namespace swgb {

const int kScoreRows[N_SCORE_ROWS] = {8, 16, 20, 25, 32, 50};

const void *score_kernel(int rows, int mode, bool fma) { return score_kernel_at<false>(rows, mode, fma); }

// The FMA-pipe diagonal add needs every substitution score minus gap_open
// to be >= 0 in the 16-bit modes (no borrow between halves).
static bool fma_add_ok(const ScoreLaunch &L) { return L.sc.mi - L.sc.go >= 0; }

int launch_score(int rows, int mode, const ScoreLaunch &L, int blocks, int threads, cudaStream_t st)
{
    const bool fma = fma_add_ok(L);
    const void *fn = L.ck_pos ? score_kernel_ck(rows, mode, fma) : score_kernel(rows, mode, fma);
    if (!fn) return SW_ERR_INVALID_ARG;
    ScoreLaunch V = L;
    void *args[] = {&V};
    if (cuda_failed(cudaLaunchKernel(fn, dim3(blocks), dim3(threads), args,
                                     score_snapshot_bytes(rows, mode, threads), st)))
        return SW_ERR_CUDA;
    count_launch();
    return launch_status();
}

// A device-planned launch of variant v = rows index * N_VMODES + mode; the
// FMA-pipe diagonal add is chosen from the scoring as for launch_score.
int launch_score_variant(int v, const ScoreLaunch &L, int blocks, cudaStream_t st)
{
    if (v < 0 || v >= N_SCORE_VARIANTS || !L.dp) return SW_ERR_INTERNAL;
    ScoreLaunch V = L;
    V.variant = v;
    return launch_score(score_rows_at(v / N_VMODES), v % N_VMODES, V, blocks, 128, st);
}

int score_variant_blocks(int v, int sm_count, int *blocks)
{
    int regs = 0, bps = 0;
    const int rc = score_kernel_regs(score_rows_at(v / N_VMODES), v % N_VMODES, &regs, &bps, 128);
    if (rc) return rc;
    if (bps < 1) return SW_ERR_INTERNAL;
    *blocks = bps * sm_count;
    return SW_OK;
}

constexpr int kAnySmem = score_snapshot_bytes(50, MODE_I16W, 128);

int launch_score_any(const ScoreLaunch &L, int blocks, cudaStream_t st)
{
    if (!L.dp || blocks < 1) return SW_ERR_INTERNAL;
    ScoreLaunch V = L;
    void *args[] = {&V};
    if (cuda_failed(cudaLaunchKernel(score_kernel_any(fma_add_ok(L)), dim3(blocks), dim3(128), args, kAnySmem, st)))
        return SW_ERR_CUDA;
    count_launch();
    return launch_status();
}

int score_any_blocks(int sm_count, int *blocks)
{
    int fewest = 0;
    for (int f = 0; f < 2; ++f) {
        const void *fn = score_kernel_any(f);
        int bps = 0;
        if (cuda_failed(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kAnySmem)) ||
            cuda_failed(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, 128, kAnySmem)))
            return SW_ERR_CUDA;
        fewest = f == 0 ? bps : std::min(fewest, bps);
    }
    if (fewest < 1) return SW_ERR_INTERNAL;
    *blocks = fewest * sm_count;
    return SW_OK;
}

// Registers and resident blocks per SM of the (rows, mode) kernels; also
// lets them take their dynamic shared memory, so it runs before any launch
// of them (both diagonal-add forms, with and without checkpoints; the grid
// follows the fewest blocks).
int score_kernel_regs(int rows, int mode, int *regs, int *max_blocks_per_sm, int threads)
{
    const int smem = score_snapshot_bytes(rows, mode, threads);
    *regs = 0;
    *max_blocks_per_sm = 0;
    for (int f = 0; f < 4; ++f) {
        const void *fn = (f & 2) ? score_kernel_ck(rows, mode, f & 1) : score_kernel(rows, mode, f & 1);
        if (!fn) return SW_ERR_INVALID_ARG;
        if (smem > 48 * 1024 &&
            cuda_failed(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)))
            return SW_ERR_CUDA;
        cudaFuncAttributes a;
        if (cuda_failed(cudaFuncGetAttributes(&a, fn))) return SW_ERR_CUDA;
        int bps = 0;
        if (cuda_failed(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, threads, smem))) return SW_ERR_CUDA;
        *regs = std::max(*regs, a.numRegs);
        *max_blocks_per_sm = f == 0 ? bps : std::min(*max_blocks_per_sm, bps);
    }
    return SW_OK;
}

}  // namespace swgb
