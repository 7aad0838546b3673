// sw_score_any.cu -- the score pass of a small batch in one launch: the bodies
// that small_body() lists, run for the variants that have classes.  255 registers,
// so 8 warps per SM whatever runs.  Most small batches have no more tasks; one of
// thousands of long reads (a task of a warp each, or two) does, and loses little:
// its plans have 20 rows or more, whose own launches hold 8 to 12 warps (4,096
// reads of 1,000 bases without a CIGAR 1.52 ms, through those launches 1.49).
#include "sw_score_kernel.cuh"

namespace swgb {

template <int R, bool FMA_ADD>
__device__ __forceinline__ void score_rows_any(const ScoreLaunch &L, int v)
{
    if constexpr (R == 20 || R == 32) {
        score_body<R, MODE_I16W, FMA_ADD, true>(L, v);
        return;
    }
    switch (v % N_VMODES) {
    case MODE_I32: score_body<R, MODE_I32, true, false>(L, v); break;
    case MODE_I16: score_body<R, MODE_I16, FMA_ADD, true>(L, v); break;
    case MODE_I16W:
        if constexpr (R == 8 || R == 16 || R == 25) {  // pipe_rows_idx
            score_body<R, MODE_I16W, FMA_ADD, true, SCORE_WARP_TASKS>(L, v);
            __syncthreads();
            score_body<R, MODE_I16W, FMA_ADD, true, SCORE_BLOCK_TASKS>(L, v);
        } else {
            score_body<R, MODE_I16W, FMA_ADD, true>(L, v);
        }
        break;
    default: score_body<R, MODE_I16S, FMA_ADD, true>(L, v); break;
    }
}

template <bool FMA_ADD>
__global__ void __launch_bounds__(128) k_score_any(const __grid_constant__ ScoreLaunch L)
{
    // (one load for the list of variants: asking for each in turn cost 24 L2
    // latencies in a row, a sixth of this kernel's time for 64 pairs)
    const int lane = threadIdx.x & 31;
    unsigned todo = __ballot_sync(0xffffffffu, lane < N_SCORE_VARIANTS && L.dp->var_n[lane] != 0);
    while (todo) {
        const int v = 31 - __clz(todo);  // longest reads first
        todo ^= 1u << v;
        switch (v / N_VMODES) {
        case 0: score_rows_any<8, FMA_ADD>(L, v); break;
        case 1: score_rows_any<16, FMA_ADD>(L, v); break;
        case 2: score_rows_any<20, FMA_ADD>(L, v); break;
        case 3: score_rows_any<25, FMA_ADD>(L, v); break;
        case 4: score_rows_any<32, FMA_ADD>(L, v); break;
        case 5: score_rows_any<50, FMA_ADD>(L, v); break;
        default: break;
        }
        __syncthreads();
    }
}

const void *score_kernel_any(bool fma)
{
    return fma ? (const void *)k_score_any<true> : (const void *)k_score_any<false>;
}

}  // namespace swgb
