// sw_score_kernel.cuh -- the Smith-Waterman score pass (score and end cell).
//
// Stage E, task iii of the paper aligns every read onto each of its extended
// CALs with Smith-Waterman.  This kernel computes, for each (read, window)
// pair, the best local-alignment score of the affine-gap recurrence
//
//   E(i,j) = max(H(i,j-1) + o, E(i,j-1) + e)
//   F(i,j) = max(H(i-1,j) + o, F(i-1,j) + e)
//   H(i,j) = max(0, H(i-1,j-1) + s(r_i, w_j), E(i,j), F(i,j))
//
// and the cell where it is first reached (smallest window index j, then
// smallest read index i).
//
// Work layout.  A group of T consecutive lanes of a warp owns one pair (int32
// mode) or two pairs (int16 modes: pair A in the low and pair B in the high
// half of every register, so each DPX instruction updates two cells).  Lane
// k of a group holds read rows k*R .. k*R+R-1 of the current row chunk in
// registers and sweeps the window columns; lane k works on column t-k at step
// t, receiving the row above its block from lane k-1 with one shuffle per
// value (a wavefront along the anti-diagonal).  The int16 modes take two
// columns per step (2(t-k) and 2(t-k)+1, four shuffles): the second column's
// rows run one row behind the first's, reading the first column's H as its
// previous column while the first reads the second's of the step before
// (two register arrays, no copies), so the two columns' F chains -- each
// row's F, max and ReLU depend on the row above -- overlap.  Reads longer than T*R are
// processed in chunks of T*R rows; the last lane of a chunk stores its bottom
// row (H+o, F per column) to global scratch for the first lane of the next
// chunk.  A warp takes floor(32/T) groups' worth of pairs at a time from a
// length-sorted list with one atomic, and loops until the list is empty.
//
// Arithmetic.  Each lane keeps per row E(i,j) and H(i,j)+o.  E and F are
// floored at 0: max(E, 0) obeys the same recurrence (because e <= 0) and
// never changes H, which is floored at 0 anyway.  The substitution score
// comes from one byte permute: per column a 4-byte table of s(x, w_j) - o for
// the four read bases x, per row a selector that picks the row's read base
// (and sign-replicates, which yields 0 or -1 -- i.e. an effective score of o
// or o-1, below zero -- for rows past the read end).  Window columns past a
// pair's end use an all-zero table, which likewise scores o.  Padded cells can
// therefore only hold values strictly below some real cell's value (o < 0), so
// they never become or tie the best cell and need no masking.
//
// (__vibmax_s16x2 is not used for the running best: the header's inline asm
// writes the max before re-reading its first operand without an early-clobber
// constraint, so with `x = __vibmax_s16x2(x, ...)` the compiler may alias the
// two and the predicates then compare the max with itself.)
//
// Best cell.  Every cell's H is turned into a key (H << TAGB) + (TAGM - r) (r = row in
// the lane's block, so equal H prefers the smaller row); a three-way-max tree
// gives the column's best key, and the lane's running best is replaced only
// when the column's H is strictly larger (so the smallest column wins).  The
// 16-bit keys need (H << TAGB) + TAGM < 32768: H <= 1022 with 5-bit row
// tags (up to 32 rows per lane), H <= 510 with 6-bit tags (up to 64 rows).
// The classifier gives this mode to pairs whose score bound is at most 510;
// with the SW_SCORE_AUTO setting larger bounds take the wide mode below.
//
// Pairs with larger possible scores (up to 32000) keep their two halves
// (MODE_I16W) but build no keys: a three-way-max tree over the rows gives
// each half's column maximum, and when a half's running best strictly rises
// the lane copies the column's R values into one of its two snapshot slots
// (shared memory, four rows per 16-byte store): the slot the other pair does
// not point to, or either when both pairs rise in the same column, so a
// column is stored once.  Each pair points to the slot of the column where
// its best was first reached, and after the chunk the best cell's row is the
// first row of that snapshot holding the best value.  This
// moves the row tracking off the ALU pipe (the kernel's limit) onto the
// shared-memory stores, so the wide mode costs the same ALU operations per
// cell as the 16-bit-key mode.  Classes whose values stay within 2047
// (MODE_I16S: reads of up to 407 bases at match 5) are a variant of it.  The
// int32 mode covers the rest.
//
// Checkpoints.  With a CIGAR to follow, the lanes whose bottom row ends a
// block of 50 to 64 read rows also store that row (H and F - o of every
// column, both pairs, two columns to a 16-byte store) in a pool from which
// the traceback recomputes one block at a time.  One store per ~800
// instructions of a step: 0.08 bytes per cell.
#pragma once
#include "sw_band.cuh"
#include "sw_device.cuh"
#include "swgb_internal.h"

namespace swgb {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t kNoCheckpoint = 0xffffffffu;

struct PairRef {
    int64_t rs, ws;  // first base of read / window
    int32_t m, n;    // lengths (m == 0: no pair)
};

__device__ __forceinline__ PairRef load_pair(const ScoreLaunch &L, const int32_t *order, int64_t n_items,
                                             int64_t item, bool on)
{
    PairRef pr{0, 0, 0, 0};
    if (on && item < n_items) {
        const int64_t p = order[item];
        const int64_t rd = L.ps.pair_read ? L.ps.pair_read[p] : p;
        pr.rs = L.ps.read_off[rd];
        pr.m = (int32_t)(L.ps.read_off[rd + 1] - pr.rs);
        pr.ws = L.ps.win_off[p];
        pr.n = (int32_t)(L.ps.win_off[p + 1] - pr.ws);
    }
    return pr;
}

// Read base codes of rows i0 .. i0+R-1 (4 bits each, 8 per word); rows past
// the read end get code 4 ("no base").
template <int R>
__device__ __forceinline__ void load_rows(const uint32_t *__restrict__ reads, const PairRef &p, int i0,
                                          uint32_t (&codes)[(R + 7) / 8])
{
#pragma unroll
    for (int q = 0; q < (R + 7) / 8; ++q) codes[q] = 0x44444444u;
#pragma unroll
    for (int q16 = 0; q16 < (R + 15) / 16; ++q16) {
        const int row = i0 + 16 * q16;
        const int cnt = min(16, p.m - row);
        if (cnt > 0) {
            uint32_t w = load_bases(reads, p.rs + row, cnt);
#pragma unroll
            for (int b = 0; b < 16; ++b) {
                const int r = 16 * q16 + b;
                if (r < R && b < cnt) {
                    uint32_t &c = codes[r / 8];
                    const int sh = 4 * (r % 8);
                    c = (c & ~(0xFu << sh)) | (((w >> (2 * b)) & 3u) << sh);
                }
            }
        }
    }
}

template <int MODE>
struct Arith;

template <>
struct Arith<MODE_I32> {
    typedef int32_t V;
    static __device__ __forceinline__ V addmax(V a, V b, V c) { return __viaddmax_s32(a, b, c); }
    static __device__ __forceinline__ V addmax_relu(V a, V b, V c) { return __viaddmax_s32_relu(a, b, c); }
    static __device__ __forceinline__ V max3(V a, V b, V c) { return __vimax3_s32(a, b, c); }
    static __device__ __forceinline__ V add(V a, V b) { return a + b; }
    static __device__ __forceinline__ V splat(int32_t x) { return x; }
};

template <>
struct Arith<MODE_I16> {
    typedef uint32_t V;
    static __device__ __forceinline__ V addmax(V a, V b, V c) { return __viaddmax_s16x2(a, b, c); }
    static __device__ __forceinline__ V addmax_relu(V a, V b, V c) { return __viaddmax_s16x2_relu(a, b, c); }
    static __device__ __forceinline__ V max3(V a, V b, V c) { return __vimax3_s16x2(a, b, c); }
    // per-half add (no carry between halves): max(a + b, -32768)
    static __device__ __forceinline__ V add(V a, V b) { return __viaddmax_s16x2(a, b, 0x80008000u); }
    static __device__ __forceinline__ V splat(int32_t x) { return ((uint32_t)(uint16_t)(int16_t)x) * 0x10001u; }
};
template <>
struct Arith<MODE_I16W> : Arith<MODE_I16> {};
template <>
struct Arith<MODE_I16S> : Arith<MODE_I16> {};

// max(a + b, 0) per half on the FMA pipe, for halves of a up to 2047 (see
// half_exact): b as a sign and magnitude, -x as 0x8000 | x.
__device__ __forceinline__ uint32_t half_add_relu(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("fma.rn.relu.f16x2 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(0x3C003C00u), "r"(b));
    return d;
}

// a * one + c on the FMA pipe; `one` is a kernel argument equal to 1, so the
// multiply-add cannot be folded into an ALU add.  With both halves of a and c
// non-negative and their sums below 32768 it is an exact per-half add.
__device__ __forceinline__ uint32_t mad_add(uint32_t a, uint32_t one, uint32_t c)
{
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(one), "r"(c));
    return d;
}

// x >> 16 on the FMA pipe (the high word of x * 65536)
__device__ __forceinline__ uint32_t hi16_fma(uint32_t x)
{
    uint32_t d;
    asm("mul.hi.u32 %0, %1, %2;" : "=r"(d) : "r"(x), "r"(0x10000u));
    return d;
}

// Rows 4q .. 4q+3 of a lane's column as one 16-byte word (rows past R: 0,
// which never equals a best value, as bests are >= 1).
template <int R, typename V>
__device__ __forceinline__ uint4 quad_of(const V (&h)[R], int q)
{
    const int r = 4 * q;
    return make_uint4((uint32_t)h[r], r + 1 < R ? (uint32_t)h[r + 1] : 0u, r + 2 < R ? (uint32_t)h[r + 2] : 0u,
                      r + 3 < R ? (uint32_t)h[r + 3] : 0u);
}

// First row of a snapshot whose half (shift 0: low, 16: high) equals best.
template <int R>
__device__ __forceinline__ int snapshot_row(const uint4 *snap, unsigned stride, uint32_t best, int shift)
{
    int row = R - 1;
    for (int q = (R + 3) / 4 - 1; q >= 0; --q) {
        const uint4 v = snap[q * stride];
        if (((v.w >> shift) & 0xFFFFu) == best) row = 4 * q + 3;
        if (((v.z >> shift) & 0xFFFFu) == best) row = 4 * q + 2;
        if (((v.y >> shift) & 0xFFFFu) == best) row = 4 * q + 1;
        if (((v.x >> shift) & 0xFFFFu) == best) row = 4 * q;
    }
    return row;
}

// Dynamic shared memory of a launch: the MODE_I16W snapshot slots.
__host__ __device__ constexpr int score_snapshot_bytes(int rows, int mode, int threads)
{
    return mode == MODE_I16W || mode == MODE_I16S ? 2 * ((rows + 3) / 4) * 16 * threads : 0;
}

// The classes of its variant that a body serves: all (their tasks are a
// warp's), those whose tasks are a warp's, or those whose tasks are a block's.
enum { SCORE_ALL, SCORE_WARP_TASKS, SCORE_BLOCK_TASKS };

// CK: checkpoints are kept for a traceback (launches without a CIGAR to
// follow run the kernels without that code: 1 % faster).
//
// Block tasks (TASKS == SCORE_BLOCK_TASKS, 32 lanes per two pairs): warp w
// takes the row chunks w, w + 4, ... of the task.  A chunk's last lane leaves
// the boundary row in the task's rows, as between the chunks of a warp's task,
// and its warp says every eight iterations how many units of two columns are
// there; the warp of the next chunk waits for them (s_prog), eight at a time,
// and requests each one iteration ahead.  A wait gives up after a limit and
// reports ST_INTERNAL.
template <int R, int MODE, bool FMA_ADD, bool CK, int TASKS = SCORE_ALL>
__device__ __forceinline__ void score_body(const ScoreLaunch &L, const int variant)
{
    typedef Arith<MODE> A;
    typedef typename A::V V;
    constexpr bool PAIR2 = MODE != MODE_I32;
    // The add of gap_open with the floor at 0 runs on the FMA pipe
    // (half_add_relu) instead of the ALU pipe, which bounds the kernel: 30,000
    // reads of 150 bases x 1-64 windows of 250 score in 7.8 ms instead of 8.6,
    // 1M pairs of 100 x 200 in 4.05 instead of 4.26.  (16-bit keys hold scores
    // up to 510, and -gap_open is at most 126.)
    constexpr bool HALF_ADD = MODE == MODE_I16 || MODE == MODE_I16S;
    constexpr int NW = (R + 7) / 8;
    // row tag in the low bits of a key: TAGM - r, so equal H prefers the
    // smaller row; 5 bits cover 32 rows, 6 bits 64
    constexpr uint32_t TAGB = R <= 32 ? 5u : 6u;
    constexpr uint32_t TAGM = (1u << TAGB) - 1u;
    static_assert(R <= 64, "row tags cover at most 64 rows");

    // column tables: s_tab[w] byte x = s(x, w) - o; s_tab[4] = 0 (padding)
    // s_tab2: two columns at once, w0 + 4 w1; 16 + w0 without the second one;
    // 20 neither
    __shared__ uint32_t s_tab[8];
    __shared__ uint2 s_tab2[21];
    const int32_t go = L.sc.go, ge = L.sc.ge;
    {
        const uint32_t mis4 = ((uint32_t)(uint8_t)(int8_t)(L.sc.mi - go)) * 0x01010101u;
        const uint32_t ma4 = ((uint32_t)(uint8_t)(int8_t)(L.sc.ma - go)) * 0x01010101u;
        auto column = [&](uint32_t w) { return prmt(mis4, ma4, 0x3210u + (4u << (4u * w))); };
        if (!PAIR2 && threadIdx.x < 8) s_tab[threadIdx.x] = threadIdx.x < 4 ? column(threadIdx.x) : 0u;
        if (PAIR2 && threadIdx.x < 21)
            s_tab2[threadIdx.x] = make_uint2(threadIdx.x < 20 ? column(threadIdx.x & 3u) : 0u,
                                             threadIdx.x < 16 ? column(threadIdx.x >> 2) : 0u);
        __syncthreads();
    }

    // MODE_I16W snapshot slots s = 0, 1: quad q of slot s at
    // snap[(s * R4 + q) * blockDim.x] (a warp's stores hit distinct banks)
    constexpr int R4 = (R + 3) / 4;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    uint4 *const snap = reinterpret_cast<uint4 *>(s_dyn) + threadIdx.x;

    const int lane = threadIdx.x & 31;
    const int64_t warp_global = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t one = (uint32_t)L.one;
    const V GO = A::splat(go), GE = A::splat(ge);
    const uint32_t GOH = 0x80008000u | ((uint32_t)(-go) * 0x10001u);
    // input already found invalid (or a plan whose shape changed): the
    // scratch may be too small for it, so do nothing
    constexpr bool PIPE = TASKS == SCORE_BLOCK_TASKS;
    const int warp = threadIdx.x >> 5;
    if constexpr (PIPE) {
        if (__syncthreads_or(*(volatile const int32_t *)L.status & ST_BAD_INPUT)) return;
    } else {
        if (*(volatile const int32_t *)L.status & ST_BAD_INPUT) return;
    }
    // block tasks: the next task, its checkpoints, each warp's best, and the
    // chunk (+ 1, upper half) and units of its boundary row that are stored
    __shared__ uint64_t s_best[PIPE ? 2 * kPipeWarps : 1], s_prog[PIPE ? kPipeWarps : 1];
    __shared__ int32_t s_base;
    __shared__ uint32_t s_ck_base;
    bool late = false;  // a wait gave up

    // One class given by the host, or every class of this launch's variant
    // in the device plan (longest reads first); the warps of the launch move
    // on to the next class as soon as the current one has no work left.
    // The class's order, count, counter and index live in shared memory, one
    // record per warp, read where they are used: held in registers across
    // the inner loops they would push the largest plans into spills.
    struct ClassCtx {
        const int32_t *order;
        int32_t *work_counter;
        int64_t n_items;
        uint8_t *bnd_warp;       // the warp's boundary slot (nullptr: one row chunk)
        int64_t bnd_group_bytes;
        int32_t cls, ci, n_cls;
        int32_t ck_rows;         // rows between the traceback's checkpoints (0: none)
        uint32_t ck_base;        // the task's first unit in the checkpoint pool
        int32_t ck_row_units, ck_n;  // units per row, rows per group
    };
    __shared__ ClassCtx s_cc[4];  // 128 threads: 4 warps
    // the wide 50-row kernels have no register to spare for a checkpoint
    // lane's place in the pool (uneven score pass 41.2 ms with 8 bytes
    // spilled, 40.8 with a shared-memory load per step)
    constexpr bool CK_SHARED = (MODE == MODE_I16W || MODE == MODE_I16S) && R >= 50;
    __shared__ uint32_t s_ck_at[CK && CK_SHARED ? 128 : 1];
    volatile ClassCtx *const cc = &s_cc[threadIdx.x >> 5];
    const bool planned = L.dp != nullptr;
    if (lane == 0) {
        cc->ci = 0;
        cc->n_cls = planned ? L.dp->var_n[variant] : 1;
    }
    __syncwarp();
    for (; cc->ci < cc->n_cls; next_index(cc->ci, lane)) {
    const int ci = cc->ci;
    int T = L.lanes, cls = L.cls;
    const int32_t *order = L.order;
    int64_t n_items = L.n_items, bnd_group_bytes = L.boundary_group_bytes;
    int32_t *work_counter = L.work_counter;
    uint8_t *bnd_base = L.boundary;
    int64_t bnd_warp_bytes = 0;  // warp stride of the boundary slots (host-given: G groups of this class)
    if (planned) {
        const DevScorePlan &dp = *L.dp;
        cls = dp.var_cls[variant][ci];
        if (TASKS != SCORE_ALL && PIPE != (dp.cls_pipe[cls] >= 0)) continue;
        T = PIPE ? 32 : dp.cls_lanes[cls];
        order = L.order + dp.cls_start[cls];
        n_items = dp.cls_count[cls];
        work_counter = L.work_counter + cls;
        bnd_group_bytes = dp.cls_bnd_bytes[cls];
        bnd_base = nullptr;
        if (PIPE) bnd_base = L.pipe + dp.cls_pipe[cls];
        if (!PIPE && bnd_group_bytes) {
            // reads in several row chunks: only warps with a boundary slot
            if (warp_global >= dp.var_bnd_warps[variant]) continue;
            bnd_base = L.boundary + dp.var_bnd_offset[variant];
            // every class of the variant uses the same warp stride, so that
            // warps working on different classes never share bytes
            bnd_warp_bytes = dp.var_bnd_slot[variant];
        }
    }
    const int G = 32 / T;
    const int g = lane / T;
    const int k = lane - g * T;
    const bool on = g < G;
    const int per_warp = G * (PAIR2 ? 2 : 1);
    if (!planned) bnd_warp_bytes = G * bnd_group_bytes;
    if (lane == 0) {
        cc->order = order;
        cc->work_counter = work_counter;
        cc->n_items = n_items;
        cc->cls = cls;
        if (CK) cc->ck_rows = planned && L.ck_pos ? L.dp->cls_ck[cls] : 0;
        cc->bnd_warp = bnd_base ? bnd_base + (PIPE ? 0 : warp_global * bnd_warp_bytes) : nullptr;
        cc->bnd_group_bytes = bnd_group_bytes;
    }
    __syncwarp();

    for (;;) {
        int base = 0;
        if constexpr (PIPE) {
            __syncthreads();
            if (threadIdx.x == 0) s_base = atomicAdd(cc->work_counter, per_warp);
            if (lane == 0) *(volatile uint64_t *)&s_prog[warp] = 0;
            __syncthreads();
            base = s_base;
        } else {
            if (lane == 0) base = atomicAdd(cc->work_counter, per_warp);
            base = __shfl_sync(FULL, base, 0);
        }
        if (base >= cc->n_items) break;

        const int64_t item = base + (int64_t)g * (PAIR2 ? 2 : 1);
        const PairRef pa = load_pair(L, cc->order, cc->n_items, item, on);
        const PairRef pb = PAIR2 ? load_pair(L, cc->order, cc->n_items, item + 1, on) : PairRef{0, 0, 0, 0};
        const int32_t mg = max(pa.m, pb.m), ng = max(pa.n, pb.n);
        const int32_t mw = __reduce_max_sync(FULL, (unsigned)mg);
        const int32_t nw = __reduce_max_sync(FULL, (unsigned)ng);
        // columns every real pair of the warp has (empty slots never feed a
        // real pair, so they do not limit the fast path)
        const int32_t na = pa.m ? pa.n : INT32_MAX, nbb = pb.m ? pb.n : INT32_MAX;
        const int32_t nmin_w = (int32_t)__reduce_min_sync(FULL, (unsigned)min(na, nbb));
        const int rows_per_chunk = T * R;
        const int chunks = (mw + rows_per_chunk - 1) / rows_per_chunk;
        const int steps = nw + T - 1;

        uint64_t bestA = 0, bestB = 0;
        if (PIPE && CK) {
            if (threadIdx.x == 0 && cc->ck_rows) {
                const int32_t rl = ((nw + 1) >> 1) + T - 1, nr = mw > 0 ? (mw - 1) / cc->ck_rows : 0;
                s_ck_base = nr ? atomicAdd(L.ck_cursor, (uint32_t)(nr * rl)) : 0u;
            }
            __syncthreads();
        }
        if (CK && cc->ck_rows) {
            if (lane == 0) {
                // (room for the columns past the window that lanes before
                // the group's last still step through)
                const int32_t rl = ((nw + 1) >> 1) + T - 1, nr = mw > 0 ? (mw - 1) / cc->ck_rows : 0;
                cc->ck_row_units = rl;
                cc->ck_n = nr;
                if (PIPE) cc->ck_base = s_ck_base;
                else cc->ck_base = nr ? atomicAdd(L.ck_cursor, (uint32_t)(G * nr * rl)) : 0u;
            }
            __syncwarp();
        }

        for (int c = PIPE ? warp : 0; c < chunks; c += PIPE ? kPipeWarps : 1) {
            const int i0 = c * rows_per_chunk + k * R;
            // per-row selectors
            uint32_t sel[R];
            {
                uint32_t ca[NW], cb[NW];
                load_rows<R>(L.ps.reads, pa, i0, ca);
                if (PAIR2) load_rows<R>(L.ps.reads, pb, i0, cb);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const uint32_t xa = (ca[r / 8] >> (4 * (r % 8))) & 0xFu;
                    if (!PAIR2) {
                        sel[r] = xa < 4u ? xa * 0x1111u + 0x8880u : 0x8888u;
                    } else {
                        const uint32_t xb = (cb[r / 8] >> (4 * (r % 8))) & 0xFu;
                        const uint32_t sa = xa < 4u ? xa * 0x11u + 0x80u : 0x88u;
                        const uint32_t sb = xb < 4u ? xb * 0x11u + 0xC4u : 0xCCu;
                        sel[r] = sa | (sb << 8);
                    }
                }
            }
            // per row: E - o and H of the previous column (E floored at o,
            // which never changes H)
            V e[R], h[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                e[r] = 0;
                h[r] = 0;
            }
            V diag_in = 0;             // H(i0-1, j-1)
            V out_h = 0, out_f = 0;    // bottom row (H, F - o) handed to the next lane
            // running best of this chunk
            uint32_t bk0 = PAIR2 && MODE == MODE_I16 ? TAGM * 0x10001u : 0u;
            uint32_t rowA = 0, rowB = 0;
            int slotA = 0, slotB = 1;  // MODE_I16W: the snapshot slot each pair points to
            int32_t jA = 0, jB = 0;
            // window stream: 2-bit codes of the next columns (up to 16)
            uint32_t wwA = 0, wwB = 0;
            const bool load_bnd = c > 0;
            const bool store_bnd = c + 1 < chunks;
            // this group's double-buffered boundary row (bytes per buffer: half)
            uint8_t *const bnd_w = cc->bnd_warp;
            const int64_t bgb = PIPE ? (int64_t)16 * nw : cc->bnd_group_bytes;
            uint8_t *const bnd = (on && bnd_w) ? bnd_w + (PIPE ? (int64_t)(base >> 1) * cc->bnd_group_bytes : g * bgb) : nullptr;
            const int64_t bnd_half = bgb / 2;
            const V *bin = load_bnd && bnd ? (const V *)(bnd + (c & 1) * bnd_half) : nullptr;
            V *bout = store_bnd && bnd ? (V *)(bnd + ((c + 1) & 1) * bnd_half) : nullptr;

            if constexpr (PAIR2) {
            // two columns per iteration: column j0 = 2(u - k) from h (its
            // previous column in h1) and column j0 + 1 from h1, interleaved
            // one row apart so that their F chains overlap
            V h1[R];
#pragma unroll
            for (int r = 0; r < R; ++r) h1[r] = 0;
            // selectors two rows to a word (prmt reads the low 16 bits; odd
            // rows are shifted down on the FMA pipe where they are used)
            uint32_t sel2[(R + 1) / 2];
#pragma unroll
            for (int r = 0; r < R; r += 2) sel2[r / 2] = sel[r] | (r + 1 < R ? sel[r + 1] << 16 : 0u);
            auto selr = [&](int r) -> uint32_t { return (r & 1) ? hi16_fma(sel2[r / 2]) : sel2[r / 2]; };
            V out_h1 = 0, out_f1 = 0;
            // a lane whose bottom row is a checkpoint stores it, two columns
            // to a 16-byte unit, from unit ck_at on
            uint32_t ck_at = kNoCheckpoint;
            if (CK) {
                if (cc->ck_rows && on) {
                    const int rows = i0 + R;
                    const int q = rows / cc->ck_rows;
                    if (q * cc->ck_rows == rows && q <= cc->ck_n)
                        ck_at = cc->ck_base + (uint32_t)((g * cc->ck_n + q - 1) * cc->ck_row_units);
                }
                if (CK_SHARED) s_ck_at[threadIdx.x] = ck_at;
            }
            // Window bases: every eight iterations each lane takes its next 16
            // columns, requested an iteration before as the two words that
            // hold them.  (When each lane asked as it got there the warp waited
            // in nearly every iteration: 30,000 reads of 150 bases x 1-64
            // windows 7.90 ms instead of 7.63, 2M uneven pairs 51.8 instead of
            // 49.1.  The loop around the cells is 130 of a step's 280
            // instructions at 8 rows per lane, 600 at 25: one branch for all
            // lanes, one 8-byte table read per pair and step.)
            uint32_t wxA = 0, wxB = 0;
            const uint32_t sh = (uint32_t)(2 * (((int)pa.ws - 2 * k) & 15)) | (uint32_t)(2 * (((int)pb.ws - 2 * k) & 15)) << 8;
            auto request = [&](int j) {
                load_columns(L.ps.wins, pa.ws, j, pa.n, wwA, wxA);
                load_columns(L.ps.wins, pb.ws, j, pb.n, wwB, wxB);
            };
            request(-2 * k);
            // iterations in which every lane has two columns of every real
            // pair: from T - 1 on, so many
            const unsigned inner = (unsigned)max(0, (nmin_w >> 1) - (T - 1));
            const int iters = (nw + 1) / 2 + T - 1;
            // block tasks: unit u of the row above, requested an iteration ahead
            uint2 in0 = make_uint2(0, 0), in1 = in0;
            auto wait_units = [&](int units) {
                if (lane == 0 && !late) {
                    const uint64_t want = ((uint64_t)c << 32) | (uint32_t)min(units, (ng + 1) >> 1);
                    volatile uint64_t *const at = &s_prog[(warp + kPipeWarps - 1) % kPipeWarps];
                    for (int spin = 0; *at < want; ++spin) {
                        if (spin >= (1 << 22)) {
                            late = true;
                            atomicOr(L.status, ST_INTERNAL);
                            break;
                        }
                        __nanosleep(40);
                    }
                }
                __threadfence_block();
                __syncwarp();
            };
            auto request_unit = [&](int u) {
                in0 = 2 * u < ng ? *(const uint2 *)&bin[4 * u] : make_uint2(0, 0);
                in1 = 2 * u + 1 < ng ? *(const uint2 *)&bin[4 * u + 2] : make_uint2(0, 0);
            };
            if (PIPE && load_bnd) {
                wait_units(9);
                if (k == 0) request_unit(0);
            }
            auto col_best = [&](const V (&hv)[R], uint32_t ck, int jj) {
                if constexpr (MODE == MODE_I16) {
                    const uint32_t nb = __vimax_s16x2_relu(bk0, ck | (TAGM * 0x10001u));
                    const uint32_t up = nb ^ bk0;
                    bk0 = nb;
                    if (up & 0xFFFFu) { rowA = ck; jA = jj; }
                    if (up > 0xFFFFu) { rowB = ck; jB = jj; }
                    return;
                }
                const uint32_t nb = __vimax_s16x2_relu(bk0, ck);
                const uint32_t up = nb ^ bk0;
                bk0 = nb;
                const bool upA = (up & 0xFFFFu) != 0, upB = up > 0xFFFFu;
                if (upA || upB) {
                    const int sl = (upA && upB) ? 0 : (upA ? (slotB ^ 1) : (slotA ^ 1));
                    uint4 *const dst = snap + sl * R4 * blockDim.x;
#pragma unroll
                    for (int q = 0; q < R4; ++q) dst[q * blockDim.x] = quad_of<R>(hv, q);
                    if (upA) { slotA = sl; jA = jj; }
                    if (upB) { slotB = sl; jB = jj; }
                }
            };
            auto add_go = [&](V u) -> V {
                if constexpr (HALF_ADD) return (V)half_add_relu((uint32_t)u, GOH);
                else return A::addmax_relu(u, GO, 0);
            };
            for (int u = 0; u < iters; ++u) {
                const int j0 = 2 * (u - k);
                V up_h0 = __shfl_up_sync(FULL, out_h, 1);
                V up_f0 = __shfl_up_sync(FULL, out_f, 1);
                V up_h1 = __shfl_up_sync(FULL, out_h1, 1);
                V up_f1 = __shfl_up_sync(FULL, out_f1, 1);
                if constexpr (PIPE) {
                    if (k == 0) {
                        up_h0 = (V)in0.x;
                        up_f0 = (V)in0.y;
                        up_h1 = (V)in1.x;
                        up_f1 = (V)in1.y;
                    }
                    if (load_bnd) {
                        if ((u & 7) == 0 && u) wait_units(u + 9);
                        if (k == 0) request_unit(u + 1);
                    }
                } else {
                    if (k == 0) up_h0 = up_f0 = up_h1 = up_f1 = 0;
                    if (load_bnd && bin && k == 0) {
                        up_h0 = j0 < ng ? bin[2 * j0] : 0;
                        up_f0 = j0 < ng ? bin[2 * j0 + 1] : 0;
                        up_h1 = j0 + 1 < ng ? bin[2 * j0 + 2] : 0;
                        up_f1 = j0 + 1 < ng ? bin[2 * j0 + 3] : 0;
                    }
                }
                if ((u & 7) == 0) {
                    wwA = __funnelshift_r(wwA, wxA, sh);
                    wwB = __funnelshift_r(wwB, wxB, sh >> 8);
                }
                uint32_t xA = wwA & 15u, xB = wwB & 15u;
                if ((unsigned)(u - (T - 1)) >= inner) {
                    xA = j0 < 0 || j0 >= pa.n ? 20u : j0 + 1 < pa.n ? xA : 16u + (xA & 3u);
                    xB = j0 < 0 || j0 >= pb.n ? 20u : j0 + 1 < pb.n ? xB : 16u + (xB & 3u);
                }
                const uint2 tA = s_tab2[xA], tB = s_tab2[xB];
                const uint32_t t0A = tA.x, t1A = tA.y, t0B = tB.x, t1B = tB.y;
                wwA >>= 4;
                wwB >>= 4;
                if ((u & 7) == 7) request(j0 + 2);
                V hu0 = up_h0, f0 = up_f0, hu1 = up_h1, f1 = up_f1;
                uint32_t ckA = 0, pkA = 0, ckB = 0, pkB = 0;
                V d0n, d1n;
                uint32_t sprev = selr(0);  // selector of the row the second column needs next
                {
                    const V s0 = (V)prmt(t0A, t0B, sprev);
                    const V s1 = (V)prmt(t1A, t1B, sprev);
                    d0n = FMA_ADD ? (V)mad_add((uint32_t)diag_in, one, (uint32_t)s0) : A::add(diag_in, s0);
                    d1n = FMA_ADD ? (V)mad_add((uint32_t)up_h0, one, (uint32_t)s1) : A::add(up_h0, s1);
                }
#pragma unroll
                for (int r = 0; r <= R; ++r) {
                    const uint32_t snext = r + 1 < R ? selr(r + 1) : 0u;
                    if (r < R) {  // column j0, row r
                        const V d = d0n;
                        e[r] = A::addmax(e[r], GE, h1[r]);
                        if (r + 1 < R) {
                            const V sn = (V)prmt(t0A, t0B, snext);
                            d0n = FMA_ADD ? (V)mad_add((uint32_t)h1[r], one, (uint32_t)sn) : A::add(h1[r], sn);
                        }
                        f0 = A::addmax(f0, GE, hu0);
                        const V hn = add_go(A::max3(d, e[r], f0));
                        h[r] = hn;
                        hu0 = hn;
                        const uint32_t k0 = MODE == MODE_I16 ? mad_add((uint32_t)hn, 1u << TAGB, (TAGM - (uint32_t)r) * 0x10001u)
                                                             : (uint32_t)hn;
                        if (r % 2 == 0) pkA = k0;
                        else ckA = r == 1 ? __vimax_s16x2_relu(pkA, k0) : __vimax3_s16x2(ckA, pkA, k0);
                    }
                    if (r >= 1) {  // column j0 + 1, row r - 1
                        const int q = r - 1;
                        const V d = d1n;
                        e[q] = A::addmax(e[q], GE, h[q]);
                        if (q + 1 < R) {
                            const V sn = (V)prmt(t1A, t1B, sprev);  // row q + 1 = r
                            d1n = FMA_ADD ? (V)mad_add((uint32_t)h[q], one, (uint32_t)sn) : A::add(h[q], sn);
                        }
                        f1 = A::addmax(f1, GE, hu1);
                        const V hn = add_go(A::max3(d, e[q], f1));
                        h1[q] = hn;
                        hu1 = hn;
                        const uint32_t k1 = MODE == MODE_I16 ? mad_add((uint32_t)hn, 1u << TAGB, (TAGM - (uint32_t)q) * 0x10001u)
                                                             : (uint32_t)hn;
                        if (q % 2 == 0) pkB = k1;
                        else ckB = q == 1 ? __vimax_s16x2_relu(pkB, k1) : __vimax3_s16x2(ckB, pkB, k1);
                    }
                    sprev = snext;
                }
                if (R % 2 == 1) {
                    ckA = R == 1 ? pkA : __vimax_s16x2_relu(ckA, pkA);
                    ckB = R == 1 ? pkB : __vimax_s16x2_relu(ckB, pkB);
                }
                diag_in = up_h1;
                out_h = hu0;
                out_f = f0;
                out_h1 = hu1;
                out_f1 = f1;
                if (CK) {
                    const uint32_t at = CK_SHARED ? *(volatile uint32_t *)&s_ck_at[threadIdx.x] : ck_at;
                    if (at != kNoCheckpoint && j0 >= 0)
                        L.ck_pool[at + ((uint32_t)j0 >> 1)] =
                            make_uint4((uint32_t)out_h, (uint32_t)out_f, (uint32_t)out_h1, (uint32_t)out_f1);
                }
                if (store_bnd && bout && k == T - 1 && j0 >= 0) {
                    if (j0 < ng) {
                        bout[2 * j0] = out_h;
                        bout[2 * j0 + 1] = out_f;
                    }
                    if (j0 + 1 < ng) {
                        bout[2 * j0 + 2] = out_h1;
                        bout[2 * j0 + 3] = out_f1;
                    }
                }
                if (PIPE && store_bnd && k == T - 1 && ((u & 7) == 7 || u + 1 == iters)) {
                    __threadfence_block();
                    *(volatile uint64_t *)&s_prog[warp] = ((uint64_t)(c + 1) << 32) | (uint32_t)max(0, u + 2 - T);
                }
                // strict improvement keeps the first column: j0 before j0 + 1
                col_best(h, ckA, j0);
                col_best(h1, ckB, j0 + 1);
            }
            } else {
            // int32: one pair per group, one column per step
            for (int t = 0; t < steps; ++t) {
                const int j = t - k;
                V up_h = __shfl_up_sync(FULL, out_h, 1);
                V up_f = __shfl_up_sync(FULL, out_f, 1);
                if (k == 0) {
                    up_h = bin && j < ng ? bin[2 * j] : 0;
                    up_f = bin && j < ng ? bin[2 * j + 1] : 0;
                }
                // column table
                uint32_t twA = 0;
                if (j >= 0) {
                    if ((j & 15) == 0) wwA = j < pa.n ? load_bases(L.ps.wins, pa.ws + j, min(16, pa.n - j)) : 0u;
                    twA = s_tab[j < pa.n ? wwA & 3u : 4u];
                    wwA >>= 2;
                }
                V hd = diag_in, hu = up_h, f = up_f;
                uint32_t ck0 = 0, pk0 = 0;  // column key, pending key
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const V s = (V)prmt(twA, 0u, sel[r]);
                    e[r] = A::addmax(e[r], GE, h[r]);
                    const V d = (V)mad_add((uint32_t)hd, one, (uint32_t)s);  // exact in int32 for any sign
                    hd = h[r];
                    f = A::addmax(f, GE, hu);
                    const V hn = A::addmax_relu(A::max3(d, e[r], f), GO, 0);
                    h[r] = hn;
                    hu = hn;
                    const uint32_t k0 = mad_add((uint32_t)hn, 1u << TAGB, TAGM - (uint32_t)r);
                    // three-way max over pairs of rows
                    if (r % 2 == 0) pk0 = k0;
                    else ck0 = r == 1 ? max(pk0, k0) : (uint32_t)__vimax3_s32((int)ck0, (int)pk0, (int)k0);
                }
                if (R % 2 == 1) ck0 = R == 1 ? pk0 : max(ck0, pk0);
                diag_in = up_h;
                out_h = h[R - 1];
                out_f = f;
                if (bout && k == T - 1 && j >= 0 && j < ng) {
                    bout[2 * j] = out_h;
                    bout[2 * j + 1] = out_f;
                }
                // strict improvement of H keeps the first (smallest) column
                if (ck0 > (bk0 | TAGM)) {
                    bk0 = ck0;
                    jA = j;
                }
            }
            }
            // fold the chunk's best into the 64-bit per-lane best
            const int rbase = c * rows_per_chunk + k * R;
            if (MODE == MODE_I32) {
                const uint32_t hb = bk0 >> TAGB;
                if (hb) bestA = max(bestA, cell_key(hb, jA, rbase + (int)TAGM - (int)(bk0 & TAGM)));
            } else if (MODE == MODE_I16) {
                const uint32_t ha = (bk0 & 0xFFFFu) >> TAGB, hb = (bk0 >> 16) >> TAGB;
                if (ha) bestA = max(bestA, cell_key(ha, jA, rbase + (int)TAGM - (int)(rowA & TAGM)));
                if (hb) bestB = max(bestB, cell_key(hb, jB, rbase + (int)TAGM - (int)((rowB >> 16) & TAGM)));
            } else {
                const uint32_t ha = bk0 & 0xFFFFu, hb = bk0 >> 16;
                const unsigned bd = blockDim.x;
                if (ha) bestA = max(bestA, cell_key(ha, jA, rbase + snapshot_row<R>(snap + slotA * R4 * bd, bd, ha, 0)));
                if (hb) bestB = max(bestB, cell_key(hb, jB, rbase + snapshot_row<R>(snap + slotB * R4 * bd, bd, hb, 16)));
            }
            __syncwarp();
        }
        // group reduction: lane k = 0 ends with the group's best
        for (int d = 1; d < T; d <<= 1) {
            const int src = (k + d < T) ? lane + d : lane;
            bestA = max(bestA, __shfl_sync(FULL, bestA, src));
            if (PAIR2) bestB = max(bestB, __shfl_sync(FULL, bestB, src));
        }
        if constexpr (PIPE) {
            if (lane == 0) {
                s_best[2 * warp] = bestA;
                s_best[2 * warp + 1] = bestB;
            }
            __syncthreads();
            if (warp) continue;
            for (int w = 1; w < kPipeWarps; ++w) {
                bestA = max(bestA, s_best[2 * w]);
                bestB = max(bestB, s_best[2 * w + 1]);
            }
        }
        // outputs, and with a traceback to follow, each pair's traceback cost
        // key (the key pass folded into this epilogue)
#pragma unroll
        for (int h2 = 0; h2 < (PAIR2 ? 2 : 1); ++h2) {
            const int64_t it = item + h2;
            int32_t tkey = -1, need32 = 0, wc = 0;
            if (on && k == 0 && it < cc->n_items) {
                const uint64_t b = h2 ? bestB : bestA;
                const int32_t p = cc->order[it];
                const uint32_t sc = key_h(b);
                const int32_t ie = sc ? key_i(b) : -1, je = sc ? key_j(b) : -1;
                L.out_score[p] = (int32_t)sc;
                L.out_end[2 * p] = ie;
                L.out_end[2 * p + 1] = je;
                if (L.tb_keys) {
                    tb_cost_key(cc->cls, (int32_t)sc, ie, je, L.sc, tkey, need32, wc);
                    L.tb_keys[p] = tkey;
                    if (CK && cc->ck_rows)
                        L.ck_pos[p] = make_uint2(cc->ck_base + (uint32_t)(g * cc->ck_n * cc->ck_row_units),
                                                 (uint32_t)(2 * cc->ck_row_units + h2));
                }
            }
            if (L.tb_keys) tb_key_atomics(tkey, cc->cls, need32, wc, L.tb_hist, L.tb_info);
        }
    }
    }  // classes
}

// Blocks per SM that the registers are held to.
constexpr int score_min_blocks(int R, int mode)
{
    return R <= 16 ? 4 : R <= 25 || (R == 32 && mode == MODE_I16) ? 3 : 2;
}

template <int R, int MODE, bool FMA_ADD, bool CK>
__global__ void __launch_bounds__(128, score_min_blocks(R, MODE)) k_score(const __grid_constant__ ScoreLaunch L)
{
    score_body<R, MODE, FMA_ADD, CK>(L, L.variant);
}

// The kernel of a mode, with or without checkpoints (the int32 mode keeps none).
template <int R, bool CK>
const void *score_kernel_of(int mode, bool fma)
{
    switch (mode) {
    case MODE_I32: return (const void *)k_score<R, MODE_I32, true, false>;
    case MODE_I16: return fma ? (const void *)k_score<R, MODE_I16, true, CK> : (const void *)k_score<R, MODE_I16, false, CK>;
    case MODE_I16W:
        return fma ? (const void *)k_score<R, MODE_I16W, true, CK> : (const void *)k_score<R, MODE_I16W, false, CK>;
    case MODE_I16S:
        return fma ? (const void *)k_score<R, MODE_I16S, true, CK> : (const void *)k_score<R, MODE_I16S, false, CK>;
    default: return nullptr;
    }
}

template <bool CK>
const void *score_kernel_at(int rows, int mode, bool fma)
{
    switch (rows) {
    case 8: return score_kernel_of<8, CK>(mode, fma);
    case 16: return score_kernel_of<16, CK>(mode, fma);
    case 20: return score_kernel_of<20, CK>(mode, fma);
    case 25: return score_kernel_of<25, CK>(mode, fma);
    case 32: return score_kernel_of<32, CK>(mode, fma);
    case 50: return score_kernel_of<50, CK>(mode, fma);
    default: return nullptr;
    }
}

// The kernels without checkpoints (sw_score.cu) and with them
// (sw_score_ck.cu): two translation units, compiled in parallel.
const void *score_kernel(int rows, int mode, bool fma);
const void *score_kernel_ck(int rows, int mode, bool fma);
// A small batch's kernel (sw_score_any.cu).
const void *score_kernel_any(bool fma);

}  // namespace swgb
