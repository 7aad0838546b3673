// sw_small.cu -- a batch of at most kSmallPairs pairs in few launches.
//
// A small call is bound by latency: the general sequence (memsets,
// classification, scan, scatter, planners, a launch per compiled variant)
// enqueues about 45 operations, most of which find nothing to do, and 64
// pairs of 100 x 150 took 390 us of which the alignment itself was a tenth.
// Here one block clears, classifies, sorts and plans the batch
// (k_small_plan), one launch holds the score kernels of every mode
// (k_score_any), one block sorts and plans the traceback (k_small_tbplan),
// and one launch serves the 16-bit traceback's wide and narrow windows; only
// the two int32 traceback launches follow.  Sorting is a bitonic sort in
// shared memory.  (The paper has no counterpart: its batches are large.)
#include "sw_classify.cuh"
#include "sw_plan.cuh"

namespace swgb {

constexpr int kSmallThreads = 1024;
static_assert(kSmallPairs <= 4096, "12 index bits below the sort key");

// Sorts s[0 .. n) ascending (n a power of two), whole block.
__device__ __forceinline__ void bitonic_sort(uint32_t *s, int n)
{
    for (int k = 2; k <= n; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < n / 2; i += blockDim.x) {
                const int a = ((i & ~(j - 1)) << 1) | (i & (j - 1)), b = a + j;
                const uint32_t x = s[a], y = s[b];
                if ((x > y) == ((a & k) == 0)) {
                    s[a] = y;
                    s[b] = x;
                }
            }
            __syncthreads();
        }
}

__device__ __forceinline__ int pow2_at_least(int n)
{
    int p = 32;
    while (p < n) p <<= 1;
    return p;
}

// keys: traceback keys to clear (nullptr: no CIGAR).  expect: the class
// counts and maxima a plan was made for, or nullptr.
__global__ void __launch_bounds__(kSmallThreads)
    k_small_plan(PairSet ps, int64_t n_reads, int n_pairs, Scoring sc, int score_setting, PlanParams pp,
                 const int32_t *__restrict__ expect, ClassInfo *info, TbClassInfo *tbinfo, int32_t *counters,
                 int32_t *tb_keys, int32_t *order, int32_t *out_score, int32_t *out_end, int32_t *cig_n,
                 DevScorePlan *splan)
{
    __shared__ uint32_t s_key[kSmallPairs];
    __shared__ ClassInfo s_info;
    for (int i = threadIdx.x; i < (int)(sizeof(ClassInfo) / 4); i += blockDim.x) ((int32_t *)&s_info)[i] = 0;
    if (threadIdx.x == 0) info->status = 0;
    for (int i = threadIdx.x; i < N_COUNTERS; i += blockDim.x) counters[i] = 0;
    if (tb_keys)
        for (int i = threadIdx.x; i < (int)(sizeof(TbClassInfo) / 4); i += blockDim.x) ((int32_t *)tbinfo)[i] = 0;
    const int np = pow2_at_least(n_pairs);
    __syncthreads();
    for (int base = 0; base < np; base += blockDim.x) {
        const int p = base + threadIdx.x;
        int32_t key = -1, cls = 0;
        int64_t m = 0, n = 0;
        if (p < n_pairs) {
            key = classify_pair(ps, n_reads, p, sc, score_setting, &info->status, out_score, out_end, cig_n, cls, m, n);
            if (tb_keys) tb_keys[p] = -1;
        }
        if (p < np) s_key[p] = key >= 0 ? ((uint32_t)key << 12) | (uint32_t)p : 0xFFFFFFFFu;
        // one set of atomics per class in the warp
        const KeyGroup g = key_group(key >= 0 ? cls : -1);
        if (key >= 0) {
            const unsigned mx_n = __reduce_max_sync(g.mask, (unsigned)n), mx_m = __reduce_max_sync(g.mask, (unsigned)m);
            const unsigned sm_n = __reduce_add_sync(g.mask, (unsigned)n);
            if (g.rank == 0) {
                atomicAdd(&s_info.count[cls], g.size);
                atomicMax(&s_info.max_n[cls], (int32_t)mx_n);
                atomicMax(&s_info.max_m[cls], (int32_t)mx_m);
                atomicAdd(&s_info.sum_n[cls], (unsigned long long)sm_n);
            }
        }
    }
    __syncthreads();
    for (int c = threadIdx.x; c < N_CLASS; c += blockDim.x) {
        info->count[c] = s_info.count[c];
        info->max_n[c] = s_info.max_n[c];
        info->max_m[c] = s_info.max_m[c];
        info->sum_n[c] = s_info.sum_n[c];
        if (expect && (s_info.count[c] != expect[c] || s_info.max_m[c] > expect[N_CLASS + c] ||
                       s_info.max_n[c] > expect[2 * N_CLASS + c]))
            atomicOr(&info->status, ST_BAD_INPUT);
    }
    bitonic_sort(s_key, np);
    for (int i = threadIdx.x; i < n_pairs; i += blockDim.x)
        if (s_key[i] != 0xFFFFFFFFu) order[i] = (int32_t)(s_key[i] & 0xFFFu);
    plan_score(&s_info, pp, splan, &info->status);
}

__global__ void __launch_bounds__(kSmallThreads)
    k_small_tbplan(const int32_t *__restrict__ tb_keys, int n_pairs, const ClassInfo *__restrict__ info,
                   const TbClassInfo *__restrict__ tbinfo, const DevScorePlan *__restrict__ splan, PlanParams pp,
                   int32_t *tb_order, DevTbPlan *tplan, int32_t *status)
{
    __shared__ uint32_t s_key[kSmallPairs];
    const int np = pow2_at_least(n_pairs);
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        const int32_t key = p < n_pairs ? tb_keys[p] : -1;
        s_key[p] = key >= 0 ? ((uint32_t)key << 12) | (uint32_t)p : 0xFFFFFFFFu;
    }
    __syncthreads();
    bitonic_sort(s_key, np);
    for (int i = threadIdx.x; i < n_pairs; i += blockDim.x)
        if (s_key[i] != 0xFFFFFFFFu) tb_order[i] = (int32_t)(s_key[i] & 0xFFFu);
    plan_tb(info, tbinfo, splan, pp, tplan, status);
}

int launch_small_plan(const PairSet &ps, int64_t n_reads, int64_t n_pairs, const Scoring &sc, int score_setting,
                      const PlanParams &pp, const int32_t *expect, ClassInfo *info, TbClassInfo *tbinfo,
                      int32_t *counters, int32_t *tb_keys, int32_t *order, int32_t *out_score, int32_t *out_end,
                      int32_t *cig_n, DevScorePlan *splan, cudaStream_t st)
{
    k_small_plan<<<1, kSmallThreads, 0, st>>>(ps, n_reads, (int)n_pairs, sc, score_setting, pp, expect, info, tbinfo,
                                              counters, tb_keys, order, out_score, out_end, cig_n, splan);
    count_launch();
    return launch_status();
}

int launch_small_tbplan(const int32_t *tb_keys, int64_t n_pairs, const ClassInfo *info, const TbClassInfo *tbinfo,
                        const DevScorePlan *splan, const PlanParams &pp, int32_t *tb_order, DevTbPlan *tplan,
                        int32_t *status, cudaStream_t st)
{
    k_small_tbplan<<<1, kSmallThreads, 0, st>>>(tb_keys, (int)n_pairs, info, tbinfo, splan, pp, tb_order, tplan,
                                                status);
    count_launch();
    return launch_status();
}

}  // namespace swgb
