// swgb_internal.h -- declarations shared by the library's translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/swgb.h"

namespace swgb {

// Status bits written by kernels (atomicOr) and read back by the host.
enum : int32_t {
    ST_BAD_INPUT = 1,
    ST_CAPACITY = 2,
    ST_INTERNAL = 4,
    ST_TIMEOUT = 8,
    ST_UNSUPPORTED = 16,
};

// The error code a call returns for a device status word: invalid input
// first, then an unsupported shape, an exhausted capacity, a device wait
// that ran out (a tensor-core kernel's bounded mbarrier wait), and internal
// errors; SW_OK when no bit is set.
inline int status_to_code(int32_t st)
{
    if (st & ST_BAD_INPUT) return SW_ERR_DEVICE_INPUT;
    if (st & ST_UNSUPPORTED) return SW_ERR_UNSUPPORTED;
    if (st & ST_CAPACITY) return SW_ERR_CAPACITY;
    if (st & ST_TIMEOUT) return SW_ERR_DEVICE_TIMEOUT;
    if (st & ST_INTERNAL) return SW_ERR_INTERNAL;
    return SW_OK;
}

// Inputs of one batch as the kernels see them (all device pointers).
struct PairSet {
    const uint32_t *reads;      // packed reads (words)
    const int64_t *read_off;    // n_reads + 1
    const int64_t *pair_read;   // n_pairs, or nullptr: pair p uses read p
    const uint32_t *wins;       // packed windows (words)
    const int64_t *win_off;     // n_pairs + 1
    const uint8_t *mask = nullptr;  // n_pairs, or nullptr: align every pair
};

struct FeatureParams {
    const uint32_t *reads;
    const int64_t *read_off;
    int64_t n_reads;
    const uint32_t *wins;
    const int64_t *win_off;
    const int64_t *cand_off;   // n_reads + 1
    uint16_t *out;             // bf16 [n_pairs][64]
};

struct Scoring {
    int32_t ma, mi, go, ge;
};

// Arithmetic of the score pass.
enum ScoreMode : int32_t {
    MODE_I32 = 0,   // one pair per lane group, int32 cells
    MODE_I16 = 1,   // two pairs per lane group in int16 halves, 16-bit keys
    MODE_I16W = 2,  // two pairs per lane group in int16 halves, 32-bit keys
    N_MODES = 3,
    // a MODE_I16W class whose values all fit half_exact(): a score variant of
    // its own, no class mode
    MODE_I16S = 3,
    N_VMODES = 4,
};

// Read-length classes: 16-base steps up to 1024, then 128-base steps.
constexpr int N_MCLASS = 64 + 56;
constexpr int N_NBUCKET = 256;       // window length / 32, clamped
constexpr int N_CLASS = N_MODES * N_MCLASS;

__host__ __device__ inline int mclass_of(int32_t m)
{
    return m <= 1024 ? (m + 15) / 16 - 1 : 64 + (m - 1024 + 127) / 128 - 1;
}
__host__ __device__ inline int32_t mclass_max(int c)
{
    return c < 64 ? 16 * (c + 1) : 1024 + 128 * (c - 64 + 1);
}

// Per-class facts the classify pass reads back to the host.
struct ClassInfo {
    int32_t count[N_CLASS];
    int32_t max_n[N_CLASS];
    int32_t max_m[N_CLASS];
    int32_t status;
    int32_t pad[3];
    unsigned long long sum_n[N_CLASS];  // window bases of the class
};

struct TbClassInfo;
struct DevScorePlan;
struct DevTbPlan;

struct ScoreLaunch {
    PairSet ps;
    Scoring sc;
    const int32_t *order;    // pair indices of this launch
    int64_t n_items;
    int32_t lanes;           // T: lanes per group
    int32_t *out_score;
    int32_t *out_end;
    uint8_t *boundary;       // per-group chunk boundaries, or nullptr
    uint8_t *pipe = nullptr; // boundary rows of block tasks
    int64_t boundary_group_bytes;
    int32_t *work_counter;
    int32_t *status;
    int32_t one = 1;         // a multiplier the compiler cannot fold
    // traceback cost keys from the epilogue (tb_keys == nullptr: none)
    int32_t cls = 0;         // the launch's class
    int32_t *tb_keys = nullptr;
    int32_t *tb_hist = nullptr;
    TbClassInfo *tb_info = nullptr;
    // row checkpoints for the traceback (classes with cls_ck in the plan):
    // the pool in 16-byte units, its cursor, and per pair (first unit, units
    // per row x 2 + half of the word the pair is in)
    uint4 *ck_pool = nullptr;
    uint32_t *ck_cursor = nullptr;
    uint2 *ck_pos = nullptr;
    // device-planned launch (dp != nullptr): the launch serves every class
    // of score variant `variant` in the plan; order is then the whole
    // sorted pair order, work_counter the base of the per-class counters and
    // boundary the base of the chunk-boundary scratch
    const DevScorePlan *dp = nullptr;
    int32_t variant = 0;
};

// What every traceback kernel needs about the batch.
struct TbParams {
    PairSet ps;
    Scoring sc;
    const int32_t *score;
    const int32_t *end;
    uint32_t *cig_ops;
    const int64_t *cig_off;
    int32_t *cig_n;
    const uint4 *ck_pool;     // row checkpoints of the score pass
    const uint2 *ck_pos;
};

// Per-class facts of the traceback sort, read back to size the slabs.
struct TbClassInfo {
    int32_t max_need[N_CLASS];  // largest slab (words) a pair of the class needs
    int32_t n_part[2][N_CLASS];    // pairs of the first two parts (tb_part_of)
    int32_t max_wcap[3][N_CLASS];  // widest chunk window of each part
};

// A persistent traceback launch: every part of traceback variant `variant`
// in the device plan.
struct TracebackLaunch {
    TbParams P;
    const int32_t *order;    // the whole traceback order (parts index into it)
    uint32_t *slab;          // base of the per-warp scratch slots
    int32_t *work_counter;   // base of the per-part counters
    int32_t *status;
    int32_t one = 1;         // a multiplier the compiler cannot fold
    const DevTbPlan *dp = nullptr;
    int32_t variant = 0;
    int32_t n_variants = 1;  // variants from `variant` on that this launch serves (of one kernel, equal slots)
};
// A launch serves the variants of one kernel: those of 16 lanes, of 8 lanes,
// then one each.
__host__ __device__ inline int tb_launch_variants(int v) { return v == 0 || v == 2 ? 2 : 1; }
__host__ __device__ inline int tb_launch_first(int v) { return v == 1 || v == 3 ? v - 1 : v; }

// Row counts compiled for the score kernels.
constexpr int N_SCORE_ROWS = 6;
extern const int kScoreRows[N_SCORE_ROWS];
constexpr int TB_ROWS = 8;
__host__ __device__ inline int score_rows_at(int i)
{
    switch (i) {
    case 0: return 8;
    case 1: return 16;
    case 2: return 20;
    case 3: return 25;
    case 4: return 32;
    default: return 50;
    }
}

// ---- device-side launch planning ----
//
// A batch is aligned by a fixed sequence of launches: the host never reads
// anything back.  One-block planner kernels turn the classification's
// per-class facts into the tables below, and every compiled kernel variant
// is launched once, persistent at full occupancy; a launch serves the
// classes (or traceback parts) its variant was given and exits at once when
// it has none.
constexpr int N_SCORE_VARIANTS = N_SCORE_ROWS * N_VMODES;  // variant = rows index * N_VMODES + mode
constexpr int N_TB16_VARIANTS = 7;                        // 16-bit traceback: T = 16 (wide windows, the rest), T = 8 (the same), T = 4, 2, 1
constexpr int TB_VAR_TILED = 7;                           // int32 traceback, one lane per pair, warp tiles
constexpr int TB_VAR_GROUPED = 8;                         // int32 traceback, T lanes per pair
constexpr int N_TB_VARIANTS = 9;
// The score launches of the general sequence fork over kScoreStreams streams.
// Launches on one stream wait for one another, and a few long reads keep a launch
// busy for milliseconds, so the row counts of the modes that long reads run in
// take turns on four of them, and the plans that reads of 75 to 800 bases get at
// one batch size (fewer rows the smaller it is) lie apart.  The fifth has the 50,
// 32 and 25 rows of the 16-bit keys: nothing waits before a batch of one length of
// short reads, and few empty launches after it.  The wide modes start first, and
// the most rows first.  Calls without a CIGAR, with every row count of a mode on
// one stream, and so: 200 reads of 1,000 to 4,000 bases 15.5 and 6.5 to 8.6 ms,
// 5,000 of 750 to 3,000 24.3 and 12.3 to 14.0, 20,000 of 75 to 800 0.95 and 0.81.
// (Where the last tasks fall decides a few batches the other way: 35,000 such
// reads with introns 1.5 and 2.1 ms.)  On eight streams the kernels take as long,
// but the device has eight queues in all, and host batches on two worker streams
// lost 6 % (14.6 to 13.7M reads/s).
constexpr int kScoreStreams = 5;
inline int score_variant_stream(int v)
{
    constexpr int8_t stream[N_SCORE_ROWS][N_VMODES] = {  // by rows; int32, 16-bit keys, wide, wide with the fp16 add
        {2, 2, 0, 0}, {3, 1, 1, 1}, {0, 3, 2, 0}, {1, 4, 3, 2}, {2, 4, 0, 1}, {3, 4, 1, 2}};
    return stream[v / N_VMODES][v % N_VMODES];
}
// The variant that is launched as number q.
inline int score_launch_order(int q)
{
    constexpr int W = MODE_I16W, S = MODE_I16S, K = MODE_I16, I = MODE_I32;
    constexpr struct { int8_t rows, mode; } order[N_SCORE_VARIANTS] = {
        {5, W}, {4, W}, {3, W}, {2, W}, {1, W}, {0, W}, {5, S}, {4, S}, {3, S}, {2, S}, {1, S}, {0, S},
        {5, K}, {3, K}, {4, K}, {2, K}, {1, K}, {0, K}, {5, I}, {4, I}, {3, I}, {2, I}, {1, I}, {0, I}};
    return order[q].rows * N_VMODES + order[q].mode;
}
__host__ __device__ inline int tb16_variant_lanes(int v) { return v < 2 ? 16 : v < 4 ? 8 : 64 >> v; }
// Rows per lane of the 16-bit kernel: with 16 lanes per two pairs, taken where
// there are too few pairs to fill the GPU, four -- a lone warp's step then
// takes 100 instructions instead of 170 while a chunk stays 64 rows.
__host__ __device__ constexpr int tb16_rows(int T) { return T == 16 ? 4 : 8; }
// Parts of a class by chunk window width: over kTbWide columns, over kTbMid,
// the rest.  A warp's scratch slot is sized for the widest window of its
// launch, and a few spliced pairs with windows of thousands of columns would
// otherwise leave room for a fraction of the warps: the wide part takes 8 or
// 16 lanes per two pairs, apart from the large narrow parts.  Over windows
// this wide the wavefront's extra steps cost little, a warp waits for the widest
// of 8 pairs rather than of 64, and a task (many blocks one after another)
// ends 7 times sooner -- the wide pairs of the 2M uneven batch took 33 ms with
// one or two lanes, most of it in the last few tasks.  The middle part
// (decoys and short introns, several times the narrow part's steps) gets its
// own number of lanes.
constexpr int kTbWide = 256, kTbMid = 64;
constexpr int kTbParts = 3;
__host__ __device__ inline int tb_part_of(int32_t wc) { return wc > kTbWide ? 0 : wc > kTbMid ? 1 : 2; }

// Lanes per two pairs of a part of a 16-bit class.  A batch too small to give a
// wave of warps tasks of 64 / T pairs spreads each two pairs over more lanes: its
// tasks (several blocks one after another) then finish sooner, which is what the
// call waits for.  The smallest run with 16 lanes in one launch; else a part takes
// lanes until its pairs make a wave, the narrow windows four at most unless that
// leaves three quarters of the warps idle (60,000 pairs of 100 x 200: 1 lane 0.58
// ms, 4 lanes 0.44; 120,000: 1 lane 0.81, 2 lanes 0.63; 16,384: 4 lanes 0.16, 16
// lanes 0.20), and long reads follow their class's count.  all, same, cnt: pairs
// of the 16-bit classes, of the part over all of them (of the last part: all),
// and of the class.
__host__ __device__ inline int tb_part_lanes(bool one_launch, int part, int64_t all, int64_t same, int64_t cnt,
                                             int32_t m_max, int32_t warps)
{
    const int64_t wave = (int64_t)warps * 64;
    int lanes = one_launch || 16 * all < wave ? 16 : part == 0 ? 8 : 1;  // (wide windows: see kTbWide)
    while (lanes < 16 && (same * lanes < (part < 2 || lanes < 4 ? wave : wave / 4) ||
                          (m_max > 512 && cnt * lanes < wave / 4)))
        lanes *= 2;
    return lanes;
}
constexpr int N_TB_PARTS = kTbParts * N_CLASS;
constexpr int kMaxPlanOverrides = 16;
constexpr int kPlanThreads = 384;                         // >= N_CLASS

// Batches of up to this many pairs (without plan overrides) take the few
// launches of sw_small.cu.
constexpr int kSmallPairs = 4096;
// Row counts that a small batch steps down through (8, 16, 25, 50), and the bodies
// in its one score launch: those, and the wide mode's 20 and 32 rows, the plans of
// most reads of 500 to 640, 800 to 1,024 and 1,600 to 2,048 bases.  (With 25 and
// 50 rows in their place 4,096 reads of 1,000 bases took 2.15 ms without a CIGAR,
// of 2,000 bases 8.1 ms; so 1.52 and 5.3.  In the int32 mode 50 rows are the
// faster: 300 reads of 7,000 bases 39.0 ms, 42.6 with 32.)
__host__ __device__ inline bool small_rows(int rows_idx) { return rows_idx != 2 && rows_idx != 4; }
__host__ __device__ inline bool small_body(int rows_idx, int vmode) { return small_rows(rows_idx) || vmode == MODE_I16W; }

// Block tasks.  A long read's two pairs in one warp take a row chunk after
// another, and a few of them leave the SMs empty: 200 reads of 1000 to 4000
// bases took 8.9 ms.  While a small batch has no more such tasks than its score
// launch has blocks, the four warps of a block take a task's chunks side by side,
// each one wavefront behind the other, with as few rows per lane as keep it at
// four chunks, 25 at most (reads over 3200 bases take more chunks).  Reads of up
// to 512 bases never do: up to there one warp takes the read in one chunk of 16
// rows or fewer.  The boundary rows of all tasks (two buffers of two values a
// column) have kPipeBytes; a class that finds no room runs as warp tasks.
constexpr int kPipeMinRead = 512, kPipeWarps = 4;
constexpr int64_t kPipeBytes = (int64_t)64 << 20;
__host__ __device__ inline bool block_task_class(int c, int32_t m_max) { return c >= N_MCLASS && m_max > kPipeMinRead; }
__host__ __device__ inline int64_t block_task_tasks(int32_t cnt) { return (cnt + 1) / 2; }
__host__ __device__ inline int64_t block_task_need(int32_t cnt, int32_t n_max) { return 16 * (int64_t)n_max * block_task_tasks(cnt); }
// Bytes of boundary rows that the block tasks of a batch take at most.
inline int64_t block_task_bytes(const ClassInfo &ci, int blocks)
{
    int64_t tasks = 0, bytes = 0;
    for (int c = 0; c < N_CLASS; ++c)
        if (ci.count[c] && block_task_class(c, ci.max_m[c])) {
            tasks += block_task_tasks(ci.count[c]);
            bytes += block_task_need(ci.count[c], ci.max_n[c]);
        }
    return tasks > blocks ? 0 : bytes < kPipeBytes ? bytes : kPipeBytes;
}
__host__ __device__ inline int pipe_rows_idx(int32_t m_max)
{
    return m_max <= kPipeWarps * 32 * 8 ? 0 : m_max <= kPipeWarps * 32 * 16 ? 1 : 3;  // 8, 16, 25 rows
}

struct PlanOverride {
    int32_t max_read_len, lanes, rows;
};

// What the planners need besides the batch's class tables (by value).
struct PlanParams {
    Scoring sc;
    int32_t n_overrides;
    PlanOverride ov[kMaxPlanOverrides];     // sorted by max_read_len
    int32_t score_warps[N_SCORE_VARIANTS];  // warps each score launch runs
    int32_t tb_warps[N_TB_VARIANTS];        // warps each traceback launch runs
    int64_t score_bnd_bytes;                // chunk-boundary scratch of the score launches
    int64_t tb_bytes;                       // traceback scratch: row checkpoints, then the warps' slots
    int64_t ck_bytes;                       // most of it that row checkpoints may take (0: none)
    int32_t allow16;                        // 16-bit traceback allowed (SW_TB_AUTO)
    int32_t small;                          // the launches of a small batch
    int32_t schedulers;                     // warp schedulers of the device
    int64_t pipe_bytes;                     // boundary rows of block tasks (small batches)
};

struct DevScorePlan {
    int32_t var_n[N_SCORE_VARIANTS];          // classes of each variant
    int32_t var_bnd_warps[N_SCORE_VARIANTS];  // warps with a boundary slot (chunked classes only)
    int64_t var_bnd_offset[N_SCORE_VARIANTS];
    int64_t var_bnd_slot[N_SCORE_VARIANTS];   // bytes of one warp's boundary slot (its largest class)
    int32_t cls_start[N_CLASS];               // first position of the class in the sorted order
    int32_t cls_count[N_CLASS];
    int32_t cls_lanes[N_CLASS];
    int32_t cls_bnd_bytes[N_CLASS];           // per group; 0 when a read fits one row chunk
    int32_t cls_ck[N_CLASS];                  // rows between checkpoints (0: none kept)
    int64_t cls_pipe[N_CLASS];                // a small batch's classes of block tasks: their boundary rows' offset, else -1
    int64_t ck_units;                         // 16-byte units of the pool the checkpoints may take
    int16_t var_cls[N_SCORE_VARIANTS][N_CLASS];  // longest reads first
};

struct TbPartPlan {
    int32_t cls, part, start, count;
    int32_t lanes, wcap;
    int64_t slab_words, bnd_ints;  // per lane (16-bit), per warp tile (tiled) or per group (grouped)
    int32_t variant;
    int32_t block_rows;            // 16-bit: rows between the class's checkpoints (0: the whole read is one block)
};

// Traceback scratch of one launch: per-warp slots from var_slot_offset on
// (words).  The 16-bit launches run at once, each in its part of what the row
// checkpoints leave; the int32 launches follow one after another, each with all
// of it.
struct DevTbPlan {
    int32_t var_n[N_TB_VARIANTS];
    int32_t var_warps[N_TB_VARIANTS];     // warps with a slot (the others exit)
    int64_t var_slot_words[N_TB_VARIANTS];
    int64_t var_slot_offset[N_TB_VARIANTS];
    int64_t split[2];                     // pairs through the 16-bit and the int32 kernels
    int16_t var_part[N_TB_VARIANTS][N_TB_PARTS];
    TbPartPlan part[N_TB_PARTS];
};

// Rows between the checkpoints of a score plan with R rows per lane: a
// multiple of R (checkpoints are bottom rows of lanes) of 50 to 64 rows,
// doubled as often as the pool's size asks for.  Narrower blocks would have
// narrower bands (a block's band allows for its own loss) but store more.
__host__ __device__ inline int ck_block_rows(int R)
{
    return R >= 50 ? R : R == 20 ? 60 : R > 16 ? 2 * R : 64;
}

// 16-byte units that the checkpoints of a class take at most: a task of
// `per_warp` pairs stores, per checkpointed row and group of two pairs, its
// widest window's columns two to a unit, and one more for each lane of a
// group but the last.  Tasks are consecutive in the order
// sorted by falling window length in buckets of 32 bases, so a task's widest
// window is at most its last pair's bucket plus the step to the task before,
// and the steps add up to the longest window once; the last bucket
// (everything past its start) is unsorted.
__host__ __device__ inline int64_t ck_class_units(int64_t cnt, int64_t sum_n, int32_t mm, int32_t mn,
                                                  int32_t lanes, int32_t block_rows)
{
    const int64_t rows = (mm - 1) / block_rows;
    const int32_t per_warp = 2 * (32 / lanes);
    const int64_t slots = cnt + per_warp;
    const int64_t cols = mn > 32 * (N_NBUCKET - 1) ? slots * mn
                                                   : sum_n + 32 * slots + (int64_t)per_warp * (mn + 32);
    return rows * (cols / 4 + slots / 2 * lanes + lanes);
}

// Score-pass arithmetic of a pair (or class) whose scores are at most hmax
// (match x min(m, n)) under a sw_set_score_mode setting: 16-bit keys up to
// 510, where 6-bit row tags leave every plan (up to 64 rows per lane) open,
// 16-bit halves without keys up to 32000, else 32-bit lanes;
// SW_SCORE_WIDE16 skips the 16-bit keys, SW_SCORE_INT32 takes 32-bit lanes.
// (Keys would fit up to 1022 with 5-bit tags, at most 32 rows per lane; the
// wide mode with 50 rows per lane measured faster on those classes.)
__host__ __device__ inline int score_mode_for(int64_t hmax, int setting)
{
    if (setting == SW_SCORE_INT32) return MODE_I32;
    if (hmax <= 510 && setting != SW_SCORE_WIDE16) return MODE_I16;
    if (hmax <= 32000) return MODE_I16W;
    return MODE_I32;
}

// Whether a 16-bit mode may take its add of gap_open with the floor at 0 as an
// fp16 multiply-add: halves 0 .. 2047 are fp16 numbers 2^-24 apart
// (subnormals and the first binade), so fp16 adds them as integers; the
// largest value is the score bound hmax less gap_open.
__host__ __device__ inline bool half_exact(int64_t hmax, const Scoring &sc) { return hmax - sc.go <= 2047; }

// The kernel mode of a class of `mode` with score bound hmax.  Reads in several
// row chunks stay in the class's mode: the variants that need boundary rows each
// take an equal part of that scratch, and one more would leave the others too
// little for the longest windows.
__host__ __device__ inline int score_vmode(int mode, int64_t hmax, const Scoring &sc, bool chunked)
{
    return mode == MODE_I16W && !chunked && half_exact(hmax, sc) ? (int)MODE_I16S : mode;
}

// Score-pass plan of a length class: lanes per group and rows per lane
// (index into score_rows_at) for reads up to m_max in `mode`, hmax the
// class's score bound.  Overrides first (sorted by max_read_len), else a
// cost model: padded rows x ~6.5 ALU operations + ~40 per lane-step (both
// measured), scaled by the share of lanes a warp leaves idle.  In the
// 16-bit-key mode more than 32 rows per lane need 6-bit row tags, which
// hold scores up to 510 only.
__host__ __device__ inline void score_plan_of(int mode, int32_t m_max, int64_t hmax, const PlanOverride *ov,
                                              int n_ov, int &lanes, int &rows_idx)
{
    const int max_rows = (mode == MODE_I16 && hmax > 510) ? 32 : 64;
    for (int i = 0; i < n_ov; ++i)
        if (m_max <= ov[i].max_read_len && ov[i].rows <= max_rows) {
            lanes = ov[i].lanes;
            rows_idx = 0;
            for (int r = 0; r < N_SCORE_ROWS; ++r)
                if (score_rows_at(r) == ov[i].rows) rows_idx = r;
            return;
        }
    // cost = chunks x T x (6.5 R + 40) / (G T / 32) = chunks x (13 R + 80) x 16 / G,
    // compared exactly as the fraction num / G (integers; the first minimum
    // over R ascending, then T ascending, wins).  Plans with one row chunk
    // need T >= ceil(m / R), and G = floor(32 / T) does not grow with T, so
    // for each R the smallest such T is the first minimum (T = 32 with one
    // chunk is never better); reads longer than 32 R take T = 32 in chunks.
    int64_t best_num = -1, best_den = 1;
    lanes = 32;
    rows_idx = 4;
    for (int ri = 0; ri < N_SCORE_ROWS; ++ri) {
        const int R = score_rows_at(ri);
        if (R > max_rows) continue;
        const int t_min = (m_max + R - 1) / R;
        const int T = t_min <= 32 ? (t_min > 0 ? t_min : 1) : 32;
        const int chunks = t_min <= 32 ? 1 : (m_max + 32 * R - 1) / (32 * R);
        const int64_t G = 32 / T;
        const int64_t num = (int64_t)chunks * (13 * R + 80) * 16;
        if (best_num < 0 || num * best_den < best_num * G) {
            best_num = num;
            best_den = G;
            lanes = T;
            rows_idx = ri;
        }
    }
}

// Traceback launch shape of one part of a class.  m_max: the class's longest read;
// max_need: the largest one-lane slab of the class (int32 kernels); wcap_in:
// the part's widest chunk window; block_rows: rows between the class's
// checkpoints (0 or m_max and more: the whole read is one block).  The 16-bit kernel
// serves every class with a 16-bit score mode unless allow16 is off, with
// lanes16 lanes per two pairs.  The int32 kernel takes one lane per pair
// where a lane's tile (every chunk at the widest window) stays small, else
// the smallest power of two with the longest read in at most 4 chunks of 8T
// rows.  Also the words one warp's scratch slot needs for this part.
constexpr int kTbChunks32 = 4;
constexpr int64_t kTiledLaneWords = 4096;
__host__ __device__ inline int64_t tb_part_shape(int mode, bool allow16, int32_t block_rows, int32_t m_max,
                                                 int64_t max_need, int32_t wcap_in, int part, const Scoring &sc,
                                                 int lanes16, TbPartPlan &t)
{
    const int64_t chunks = (m_max + TB_ROWS - 1) / TB_ROWS;
    int32_t wcap = wcap_in > 1 ? wcap_in : 1;
    t.block_rows = 0;
    if (allow16 && mode != MODE_I32) {
        const int T = lanes16;
        const int64_t rows = block_rows && block_rows < m_max ? block_rows : m_max;
        const int rc = T * tb16_rows(T);
        const int64_t chunks_t = (rows + rc - 1) / rc;
        // a block entered inside an insertion run does not pay for opening
        // it, so its band may be a few columns wider than the whole pair's;
        // windows start at multiples of four columns
        wcap = (wcap + (sc.ge - sc.go) / (sc.ma - sc.ge) + 2 + (rc - 8) + 3 + 3) / 4 * 4;
        const int64_t s4 = (wcap + T - 1 + 3) / 4;
        t.lanes = T;
        t.wcap = wcap;
        t.block_rows = block_rows;
        t.slab_words = chunks_t * s4 * tb16_rows(T);     // per lane
        t.bnd_ints = (int64_t)(32 / T) * 2 * (wcap + 8);  // per warp: one row
        t.variant = T == 16 ? (part ? 1 : 0) : T == 8 ? (part ? 3 : 2) : T == 4 ? 4 : T == 2 ? 5 : 6;
        return ((32 * t.slab_words + 63) & ~(int64_t)63) + t.bnd_ints;
    }
    int T = 1;
    while (T < 32 && (int64_t)T * 8 * kTbChunks32 < m_max) T *= 2;
    const bool tiled = chunks * wcap <= kTiledLaneWords;
    if (tiled) T = 1;
    t.lanes = T;
    t.wcap = wcap;
    if (tiled) {
        t.slab_words = chunks * wcap;                  // per lane
        t.bnd_ints = chunks > 1 ? (int64_t)4 * wcap : 0;
        t.variant = TB_VAR_TILED;
        return 32 * (t.slab_words + t.bnd_ints);
    }
    const int64_t chunks_t = (m_max + 8 * T - 1) / (8 * T);
    const int64_t wcap_t = wcap + 8 * (T - 1);
    t.slab_words = T == 1 ? (max_need > 1 ? max_need : 1) : chunks_t * wcap_t * T;  // per group
    t.bnd_ints = chunks_t > 1 ? (int64_t)4 * wcap_t : 0;
    t.variant = TB_VAR_GROUPED;
    return (int64_t)(32 / T) * (t.slab_words + t.bnd_ints);
}

// score_setting: the sw_set_score_mode value (SW_SCORE_INT32: every pair in
// the int32 mode; SW_SCORE_WIDE16: no 16-bit keys; else the narrowest
// mode its score bound allows)
int launch_classify(const PairSet &ps, int64_t n_reads, int64_t n_pairs, Scoring sc, int score_setting,
                    int32_t *keys, int32_t *hist, int32_t *bucket_start, int32_t *cursor,
                    ClassInfo *info, int32_t *order, int32_t *out_score, int32_t *out_end,
                    int32_t *cig_n, cudaStream_t st);
int launch_score(int rows, int mode, const ScoreLaunch &L, int blocks, int threads, cudaStream_t st);
int score_kernel_regs(int rows, int mode, int *regs, int *max_blocks_per_sm, int threads);
int launch_check_counts(const ClassInfo *info, const int32_t *expect, int32_t *status, cudaStream_t st);
int launch_plan_score(const ClassInfo *info, const PlanParams &pp, DevScorePlan *out, int32_t *status,
                      cudaStream_t st);
int launch_plan_tb(const ClassInfo *info, const TbClassInfo *ti, const DevScorePlan *sp, const PlanParams &pp,
                   DevTbPlan *out, int32_t *status, cudaStream_t st);
// One persistent launch of score variant v (rows index * N_VMODES + mode) at
// full occupancy; its grid (blocks) comes from score_variant_blocks.
int launch_score_variant(int v, const ScoreLaunch &L, int blocks, cudaStream_t st);
int score_variant_blocks(int v, int sm_count, int *blocks);
// (every variant from v on of its kernel)
int launch_traceback_variant(int v, bool fma, const TracebackLaunch &L, int blocks, cudaStream_t st);
// The one score launch of a small batch: every class of every variant.
int launch_score_any(const ScoreLaunch &L, int blocks, cudaStream_t st);
int score_any_blocks(int sm_count, int *blocks);
int launch_small_plan(const PairSet &ps, int64_t n_reads, int64_t n_pairs, const Scoring &sc, int score_setting,
                      const PlanParams &pp, const int32_t *expect, ClassInfo *info, TbClassInfo *tbinfo,
                      int32_t *counters, int32_t *tb_keys, int32_t *order, int32_t *out_score, int32_t *out_end,
                      int32_t *cig_n, DevScorePlan *splan, cudaStream_t st);
int launch_small_tbplan(const int32_t *tb_keys, int64_t n_pairs, const ClassInfo *info, const TbClassInfo *tbinfo,
                        const DevScorePlan *splan, const PlanParams &pp, int32_t *tb_order, DevTbPlan *tplan,
                        int32_t *status, cudaStream_t st);
int traceback_variant_blocks(int v, int sm_count, int *blocks);
// Work counters of one batch: score (per class), traceback (per part), and
// the checkpoint pool's cursor.
constexpr int CTR_TB = N_CLASS, CTR_CK = CTR_TB + N_TB_PARTS;
constexpr int N_COUNTERS = CTR_CK + 1;
int launch_scan_scatter(const int32_t *keys, int64_t n_pairs, const int32_t *class_count, int32_t *hist,
                        int32_t *bucket_start, int32_t *cursor, int32_t *order, cudaStream_t st);

int launch_features(const FeatureParams &P, int sm_count, cudaStream_t st);
int64_t mlp_floats();
int launch_mlp_init(float *model, uint64_t seed, cudaStream_t st);
int launch_mlp_refresh(float *model, cudaStream_t st);
int launch_mlp_forward(const float *model, const uint16_t *feat, int64_t n, float *out, int sm_count,
                       cudaStream_t st);
int launch_mlp_grad(float *model, const uint16_t *feat, const float *target, const int32_t *idx, int64_t n,
                    int sm_count, cudaStream_t st);
int launch_mlp_adam(float *model, float lr, int32_t step, cudaStream_t st);
// The filter's selection rules, by value in the kernel's parameters.
struct SelectRules {
    int32_t n;
    int32_t max_len[SW_FILTER_MAX_RULES];
    int32_t k[SW_FILTER_MAX_RULES];
    float tau[SW_FILTER_MAX_RULES];
    float delta[SW_FILTER_MAX_RULES];
};
int launch_select(const float *pred, const int64_t *cand_off, const int64_t *read_off, int64_t n_reads,
                  const SelectRules &rules, uint8_t *mask, cudaStream_t st);
int launch_best_per_read(const int32_t *score, const int64_t *cand_off, int64_t n_reads, const uint8_t *mask,
                         int32_t *best, int32_t *best_cand, cudaStream_t st);

int launch_top_hits(const int32_t *score, const int64_t *cand_off, int64_t n_reads, const uint8_t *mask, int32_t *best,
                    int32_t *best_cand, int32_t *second, int32_t *mapq, cudaStream_t st);
int launch_records(const int32_t *score, const int32_t *end, const sw_cigar_t &cig, int64_t n_pairs,
                   const int32_t *chrom, const int64_t *pos, const int8_t *strand, int32_t min_score,
                   sw_record_t *out, int64_t *out_count, int32_t *blk_count, int64_t *blk_off, cudaStream_t st);
int launch_junctions(const uint32_t *wins, const int64_t *win_off, const int32_t *score, const int32_t *end,
                     const sw_cigar_t &cig, int64_t n_pairs, const int32_t *chrom, const int64_t *pos,
                     int32_t min_score, int32_t min_intron, uint64_t *table, int64_t capacity, int32_t *status,
                     cudaStream_t st);
int launch_table_clear(uint64_t *table, int64_t capacity, cudaStream_t st);
int launch_table_export(const uint64_t *table, int64_t capacity, sw_junction_t *out, int64_t max_out,
                        int64_t *out_count, cudaStream_t st);

int launch_cigar_to_host(const uint32_t *ops, const int64_t *off, const int32_t *n_ops, int64_t n_pairs,
                         uint32_t *host_ops, cudaStream_t st);

int launch_cap_offsets(const int64_t *read_off, int64_t n_pairs, int64_t *cig_off, int64_t *blk, cudaStream_t st);
int launch_cap_offsets_indexed(const int64_t *read_off, const int64_t *pair_read, int64_t n_pairs, int64_t *cig_off,
                               int64_t *blk, cudaStream_t st);
int launch_dense_cigar(const uint32_t *ops, const int64_t *off, const int32_t *n_ops, int64_t n_pairs,
                       int64_t *doff, uint32_t *dense, int64_t dense_cap, int64_t *blk, cudaStream_t st);

int launch_mlp_forward_tc(const float *model, const uint16_t *feat, int64_t n, float *out, int sm_count,
                          int32_t *status, cudaStream_t st);
// The gradient on the tensor cores: one partial per CTA (partial: that many
// x GRAD_PART floats), then their sum in CTA order into the model's gradient.
int mlp_grad_tc_parts(int64_t n, int sm_count);
int launch_mlp_grad_tc(float *model, const uint16_t *feat, const float *target, const int32_t *idx, int64_t n,
                       int sm_count, float *partial, int32_t *status, cudaStream_t st);
// Scratch of sw_mlp_grad on this stream (grown on demand).
int grad_scratch(cudaStream_t st, size_t bytes, float **ptr);
// A device status word for calls outside the alignment path: cleared on
// `st`, and the word sw_sync_status reads until the next call sets another.
int aux_status_word(cudaStream_t st, int32_t **status);
int filter_scratch(cudaStream_t st, size_t bytes, uint8_t **ptr);
int stream_status_word(cudaStream_t st, int32_t **status);
int launch_or_status(int32_t *dst, const int32_t *src, cudaStream_t st);

// Layout of the filter's model buffer (floats): parameters, Adam moments,
// gradient, step, then bf16 copies of W1 and W2 transposed (K-major).
constexpr int64_t MD_W1 = 0, MD_B1 = 16384, MD_W2 = 16640, MD_B2 = 33024, MD_W3 = 33088, MD_B3 = 33152;
constexpr int64_t MD_NP = 33153;
constexpr int64_t MD_M = MD_NP, MD_V = 2 * MD_NP, MD_G = 3 * MD_NP, MD_STEP = 4 * MD_NP;
constexpr int64_t MD_W1T = 132616;          // bf16 [256][64], 16-byte aligned
constexpr int64_t MD_W2T = MD_W1T + 8192;   // bf16 [64][256]
constexpr int64_t MD_TOTAL = MD_W2T + 8192;
constexpr int64_t GRAD_PART = (MD_NP + 3) / 4 * 4;  // one CTA's partial gradient, 16-byte aligned

void count_launch(int n = 1);

// The CUDA error behind the last SW_ERR_CUDA of this host thread.
void note_cuda_error(cudaError_t e);
inline bool cuda_failed(cudaError_t e)
{
    if (e == cudaSuccess) return false;
    note_cuda_error(e);
    return true;
}
inline int launch_status() { return cuda_failed(cudaGetLastError()) ? SW_ERR_CUDA : SW_OK; }

// Exclusive scan of int32 values v[0 .. n) into out[0 .. n] (out[n] = the
// total); blk holds (n + 255) / 256 + 1 int64 words.
int launch_scan_i32(const int32_t *v, int64_t n, int64_t *out, int64_t *blk, cudaStream_t st);

// ---- seeding (reads to candidate windows) ----
struct SeedKParams {
    int32_t k, stride, phase, max_hits, merge_dist, min_cal_len, flank, max_intron, max_window;
};
struct SeedOutPtrs {
    int64_t *start;
    int32_t *length;
    int32_t *chrom;
    int64_t *pos;
    int8_t *strand;
    int64_t *pair_read;
    int64_t *cand_offsets;
    int64_t *count;
};
int seed_count_per_read(int m, const SeedKParams &p);
int launch_index_build(const uint32_t *genome, int64_t n_bases, const int64_t *chrom_off, int n_chrom, int k,
                       uint32_t *table, uint32_t *positions, int64_t *out_n, uint32_t *blk, int sm_count,
                       int32_t *status, cudaStream_t st);
size_t seed_scratch_bytes(int64_t n_reads, int64_t capacity);
int launch_seed_windows(const uint32_t *reads, const int64_t *roff, int64_t n_reads, const uint32_t *table,
                        const uint32_t *positions, const int64_t *chrom_off, int n_chrom, const SeedKParams &p,
                        int max_read, int block_hits, SeedOutPtrs out, int64_t capacity, uint8_t *scratch,
                        int64_t *stats_host, int sm_count, int32_t *status, cudaStream_t st);
int launch_extract_windows(const uint32_t *genome, int64_t n_bases, const int64_t *start, const int32_t *len,
                           int64_t n, uint32_t *dst, int64_t cap_bases, int64_t *woff, int64_t *blk, int sm_count,
                           int32_t *status, cudaStream_t st);
int launch_two_strands(const uint32_t *reads, const int64_t *roff, int64_t n, uint32_t *dst, int64_t cap_bases,
                       int64_t *doff, int sm_count, int32_t *status, cudaStream_t st);

}  // namespace swgb
