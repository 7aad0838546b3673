// sw_traceback.cu -- CIGAR of the best local alignment of each pair.
//
// The paper's Stage E, task iii returns the alignment itself, not only its
// score; downstream, long runs of deletions in it mark splice junctions.
// The score pass keeps no traceback bits.  This pass recomputes the DP exactly
// over a region that provably holds every optimal alignment ending at the end
// cell (i_end, j_end), and walks back through it: the 16-bit kernel (further
// down) block by block from the score pass's row checkpoints, the int32
// kernel over the whole read's band.
//
// The band of the int32 kernel.  Any alignment with this score that ends on read row i_end
// holds at most i_end+1 aligned read bases, each worth at most `match`, and
// with o <= e <= 0 one gap run is the cheapest way to spend gap bases, so
//   deletions  D <= (match (i_end+1) + o - score) / (-e) + 1
//   insertions I <= (match (i_end+1) + o - e - score) / (match - e).
// Walking back from the end cell, a deletion lowers the diagonal d = j - i by
// one and an insertion raises it by one, so every optimal path stays in the
// band  j_end - i_end - D <= j - i <= j_end - i_end + I,  rows 0..i_end.
// Cells outside the band are treated as unreachable (H = 0, E = F = -inf);
// that can only lower recomputed values, and cells on optimal paths keep
// theirs, so every comparison of the walk comes out as in the full matrix.
//
// Layout.  A group of T lanes owns one pair; lane k holds 8 rows of a chunk of
// 8T rows and sweeps the chunk's band window of columns with a one-step
// wavefront (shuffles pass the bottom row down); the chunk's last lane hands
// its bottom row to the next chunk through a double-buffered scratch row.
// Each cell stores 4 bits -- bits 0-1 the source of H (0: H == 0, 1: diagonal,
// 2: E, 3: F, in that order of preference), bit 2 "E opens here"
// (E == H(i,j-1) + o), bit 3 "F opens here" -- one 32-bit word per lane and
// column, in a per-group slab.  The group's first lane then walks back from
// the end cell, writes the runs reversed into the pair's CSR slot and
// reverses them in place.
//
// Scheduling.  The score pass's epilogue gives every pair a cost key (its
// chunk window), a counting sort orders each length class by it so a warp's
// groups sweep similar windows, and pairs with wide windows form a part of
// their own with larger slabs.  A device
// planner (sw_devplan.cu) sizes every part and assigns it to one of the
// persistent launches below; each warp of a launch owns one scratch slot,
// sized for the largest part of its launch.
#include <algorithm>

#include "sw_band.cuh"
#include "sw_device.cuh"
#include "swgb_internal.h"

namespace swgb {

constexpr unsigned FULLMASK = 0xffffffffu;

struct TbPair {
    int64_t rs, ws;
    int32_t m, n, score, ie, je;
    int32_t jlo, W, rows;   // rectangle: window columns jlo .. jlo+W-1, rows 0..rows-1
    int32_t a, b;           // band in rectangle columns: row i spans [i + a, i + b]
    int32_t p;
};

__device__ __forceinline__ TbPair tb_pair(const TbParams &P, int32_t p, int32_t *status)
{
    TbPair q{};
    q.p = p;
    q.ie = -1;
    q.je = -1;
    if (p < 0) return q;
    const int64_t rd = P.ps.pair_read ? P.ps.pair_read[p] : p;
    q.rs = P.ps.read_off[rd];
    q.m = (int32_t)(P.ps.read_off[rd + 1] - q.rs);
    q.ws = P.ps.win_off[p];
    q.n = (int32_t)(P.ps.win_off[p + 1] - q.ws);
    q.score = P.score[p];
    if (q.score <= 0) return q;
    q.ie = P.end[2 * p];
    q.je = P.end[2 * p + 1];
    if (q.ie < 0 || q.ie >= q.m || q.je < 0 || q.je >= q.n || q.score > P.sc.ma * min(q.m, q.n)) {
        // an end cell outside the pair: never walk it
        if (status) atomicOr(status, ST_INTERNAL);
        q.score = 0;
        return q;
    }
    const Band bd = band_of(q.score, q.ie, q.je, P.sc);
    q.jlo = bd.jlo;
    q.W = bd.W;
    q.rows = bd.rows;
    q.a = bd.a;
    q.b = bd.b;
    return q;
}

// Run-length writer that emits runs in reverse order into a CSR slot.
struct RevCigar {
    uint32_t *out;
    int64_t cap;
    int32_t n;
    uint32_t op;
    int32_t len;
    bool overflow;
    __device__ void push(uint32_t o, int32_t l)
    {
        if (l <= 0) return;
        if (len > 0 && o == op) {
            len += l;
            return;
        }
        flush();
        op = o;
        len = l;
    }
    __device__ void flush()
    {
        if (len > 0) {
            if (n < cap) out[n] = ((uint32_t)len << 4) | op;
            else overflow = true;
            ++n;
        }
        len = 0;
    }
};

__device__ __forceinline__ int64_t lmin(int64_t a, int64_t b) { return a < b ? a : b; }

// Band window of chunk c (rows c*rc .. c*rc+rc-1) in rectangle columns.
__device__ __forceinline__ void chunk_window(const TbPair &q, int c, int rc, int &lo, int &hi)
{
    lo = max(0, c * rc + q.a);
    hi = min(q.W - 1, c * rc + rc - 1 + q.b);
}

// Slab words a pair needs with T lanes: sum over chunks of window x T.
__device__ __forceinline__ int64_t slab_need(const TbPair &q, int T)
{
    if (q.score <= 0) return 0;
    const int rc = T * TB_ROWS;
    const int chunks = (q.rows + rc - 1) / rc;
    const int wcap = min(q.W, rc - 1 + (q.b - q.a) + 1);
    return (int64_t)chunks * wcap * T;
}

// TILED (one lane per pair only): the warp's slabs and boundary rows are
// interleaved lane-minor -- word (chunk c, column jl) of lane l at
// [(c * WCAP + jl) * 32 + l] -- so that, all lanes being at the same chunk
// and column at every step, each store instruction writes one full line.
// Otherwise every group owns a packed slab of its chunks' windows.
template <bool TILED>
__global__ void __launch_bounds__(128) k_traceback(const TracebackLaunch L)
{
    const TbParams &P = L.P;
    // column tables: s_tab[w] byte x = s(x, w) - o
    __shared__ uint32_t s_tab[4];
    {
        const uint32_t mis4 = ((uint32_t)(uint8_t)(int8_t)(P.sc.mi - P.sc.go)) * 0x01010101u;
        const uint32_t ma4 = ((uint32_t)(uint8_t)(int8_t)(P.sc.ma - P.sc.go)) * 0x01010101u;
        if (threadIdx.x < 4) s_tab[threadIdx.x] = prmt(mis4, ma4, 0x3210u + (4u << (4u * threadIdx.x)));
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int64_t warp_global = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int32_t go = P.sc.go, ge = P.sc.ge;
    const DevTbPlan &dp = *L.dp;
    const int v = L.variant;
    // warps without a scratch slot, and input already found invalid
    if (warp_global >= dp.var_warps[v]) return;
    // (an unsupported size means some pairs were not scored, so the
    // traceback order is incomplete: do nothing)
    if (*(volatile const int32_t *)L.status & (ST_BAD_INPUT | ST_UNSUPPORTED)) return;
    uint32_t *const slot = L.slab + dp.var_slot_offset[v] + warp_global * dp.var_slot_words[v];

    for (int pi = 0; pi < dp.var_n[v]; ++pi) {
    const TbPartPlan &tp = dp.part[dp.var_part[v][pi]];
    const int T = tp.lanes;
    const int G = 32 / T;
    const int g = lane / T;
    const int k = lane - g * T;
    const bool on = g < G;
    const int rc = T * TB_ROWS;
    const int WCAP = tp.wcap;
    const int64_t slab_words = tp.slab_words, bnd_ints = tp.bnd_ints;
    const int32_t *const order = L.order + tp.start;
    const int64_t n_items = tp.count;
    int32_t *const counter = L.work_counter + kTbParts * tp.cls + tp.part;
    // the warp's slot: TILED -> one tile indexed with the lane, then the
    // boundary rows; else every group's slab, then every group's boundary row
    uint32_t *slab = !on ? nullptr : TILED ? slot : slot + g * slab_words;
    int32_t *bnd = !on ? nullptr
                       : TILED ? (int32_t *)(slot + 32 * slab_words)
                               : (int32_t *)(slot + G * slab_words + g * bnd_ints);
    const int64_t bnd_half = TILED ? 32 * (bnd_ints / 2) : bnd_ints / 2;

    for (;;) {
        int base = 0;
        if (lane == 0) base = atomicAdd(counter, G);
        base = __shfl_sync(FULLMASK, base, 0);
        if (base >= n_items) break;
        const int64_t item = base + g;
        const int32_t p = (on && item < n_items) ? order[item] : -1;
        TbPair q = tb_pair(P, p, L.status);
        const bool over = TILED ? (q.rows > (slab_words / max(WCAP, 1)) * rc ||
                                   min(q.W, rc + (q.b - q.a)) > WCAP)
                                : (slab_need(q, T) > slab_words ||
                                   (q.rows > rc && 4 * (int64_t)min(q.W, rc + (q.b - q.a)) > bnd_ints));
        if (q.score > 0 && over) {
            // the launch was sized from the class maxima; never overrun a slab
            // or a boundary row
            atomicOr(L.status, ST_INTERNAL);
            q.score = 0;
            q.rows = 0;
        }
        const int32_t rows_w = __reduce_max_sync(FULLMASK, (unsigned)(q.score > 0 ? q.rows : 0));
        const int chunks = (rows_w + rc - 1) / rc;
        const int wcap = q.score > 0 ? min(q.W, rc - 1 + (q.b - q.a) + 1) : 0;
        int64_t slab_off = 0;  // words before chunk c in this group's slab

        int prev_lo = 0, prev_hi = -1;
        for (int c = 0; c < chunks; ++c) {
            int lo = 0, hi = -1;
            if (q.score > 0 && c * rc < q.rows) chunk_window(q, c, rc, lo, hi);
            const int width = hi - lo + 1;
            const int steps = __reduce_max_sync(FULLMASK, (unsigned)max(width, 0)) + T - 1;
            const int i0 = c * rc + k * TB_ROWS;
            // per-row selectors into the column table (sign-extended byte);
            // rows past the end row are never read by the walk
            uint32_t sel[TB_ROWS];
            {
                uint32_t codes = 0x44444444u;  // 4 bits per row, 4 = no base
                const int cnt = min(TB_ROWS, q.rows - i0);
                if (q.score > 0 && cnt > 0) {
                    const uint32_t w = load_bases(P.ps.reads, q.rs + i0, cnt);
#pragma unroll
                    for (int r = 0; r < TB_ROWS; ++r)
                        if (r < cnt) codes = (codes & ~(0xFu << (4 * r))) | (((w >> (2 * r)) & 3u) << (4 * r));
                }
#pragma unroll
                for (int r = 0; r < TB_ROWS; ++r) {
                    const uint32_t x = (codes >> (4 * r)) & 0xFu;
                    sel[r] = x < 4u ? x * 0x1111u + 0x8880u : 0x8888u;
                }
            }
            // per row: E - o and H of the previous column.  E - o is floored
            // at 0: since H >= 0 the floor never changes max(H + o, E + e) or
            // which of the two is larger, so E, F and the open bits the walk
            // reads are exact.
            int32_t E[TB_ROWS], Hp[TB_ROWS];
#pragma unroll
            for (int r = 0; r < TB_ROWS; ++r) {
                E[r] = 0;
                Hp[r] = 0;
            }
            // boundary rows are indexed relative to the writing chunk's window
            const int32_t *bin = (bnd && c > 0) ? bnd + (c & 1) * bnd_half : nullptr;
            int32_t *bout = (bnd && c + 1 < chunks) ? bnd + ((c + 1) & 1) * bnd_half : nullptr;
            // diagonal into the chunk's first column: the previous chunk's
            // bottom row one column to the left, if it computed it
            int32_t diag_in = 0;
            // boundary element (column x of the writing chunk, value v)
            auto bidx = [&](int x, int v) -> int64_t { return TILED ? ((int64_t)x * 2 + v) * 32 + lane : 2 * x + v; };
            if (k == 0 && bin && lo - 1 >= prev_lo && lo - 1 <= prev_hi) diag_in = bin[bidx(lo - 1 - prev_lo, 0)];
            int32_t out_h = 0, out_f = 0;
            // the first lane reads the row above from the previous chunk two
            // columns ahead, so the loads are in flight while columns compute
            int32_t nb_h = 0, nb_f = 0, nc_h = 0, nc_f = 0;
            if (k == 0 && bin) {
                if (lo >= prev_lo && lo <= prev_hi) {
                    nb_h = bin[bidx(lo - prev_lo, 0)];
                    nb_f = bin[bidx(lo - prev_lo, 1)];
                }
                if (lo + 1 >= prev_lo && lo + 1 <= prev_hi) {
                    nc_h = bin[bidx(lo + 1 - prev_lo, 0)];
                    nc_f = bin[bidx(lo + 1 - prev_lo, 1)];
                }
            }
            // window bases: ww holds the current word's remaining bases, wn the
            // next 16-base word (requested 16 columns before it is needed)
            const int64_t abs_lo = q.ws + q.jlo + lo, abs_hi = q.ws + q.jlo + hi;
            uint32_t ww = 0, wn = 0;
            int64_t apos = abs_lo;
            if (width > 0) {
                const int64_t a1 = (abs_lo & ~(int64_t)15) + 16;
                ww = load_bases(P.ps.wins, abs_lo, (int)lmin(a1 - abs_lo, abs_hi - abs_lo + 1));
                wn = a1 <= abs_hi ? load_bases(P.ps.wins, a1, (int)lmin(16, abs_hi - a1 + 1)) : 0u;
            }

            for (int t = 0; t < steps; ++t) {
                const int jl = t - k;       // column within the window
                const int jj = lo + jl;     // rectangle column
                int32_t up_h = __shfl_up_sync(FULLMASK, out_h, 1);
                int32_t up_f = __shfl_up_sync(FULLMASK, out_f, 1);
                if (k == 0) {
                    up_h = nb_h;
                    up_f = nb_f;
                    nb_h = nc_h;
                    nb_f = nc_f;
                    const int nx = jj + 2;
                    if (bin && nx >= prev_lo && nx <= prev_hi) {
                        nc_h = bin[bidx(nx - prev_lo, 0)];
                        nc_f = bin[bidx(nx - prev_lo, 1)];
                    } else {
                        nc_h = 0;
                        nc_f = 0;
                    }
                }
                if (jl >= 0 && jl < width) {
                    const uint32_t tw = s_tab[ww & 3u];
                    ww >>= 2;
                    if (((++apos) & 15) == 0) {
                        ww = wn;
                        const int64_t a2 = apos + 16;
                        wn = a2 <= abs_hi ? load_bases(P.ps.wins, a2, (int)lmin(16, abs_hi - a2 + 1)) : 0u;
                    }
                    int32_t d0 = diag_in, hu = up_h, f = up_f;
                    uint32_t word = 0;
#pragma unroll
                    for (int r = 0; r < TB_ROWS; ++r) {
                        const int32_t sp = (int32_t)prmt(tw, 0u, sel[r]);  // s - o
                        const int32_t eext = E[r] + ge;
                        const int32_t e = max(Hp[r], eext);
                        const int32_t fext = f + ge;
                        f = max(hu, fext);
                        const int32_t d = d0 + sp;
                        const int32_t u = __vimax3_s32(d, e, f);
                        const int32_t h = max(u + go, 0);
                        uint32_t code = h == 0 ? 0u : (u == d ? 1u : (u == e ? 2u : 3u));
                        code |= (Hp[r] >= eext ? 4u : 0u) | (hu >= fext ? 8u : 0u);
                        word |= code << (4 * r);
                        d0 = Hp[r];
                        Hp[r] = h;
                        E[r] = e;
                        hu = h;
                    }
                    if (TILED) slab[((int64_t)c * WCAP + jl) * 32 + lane] = word;
                    else slab[slab_off + (int64_t)jl * T + k] = word;
                    out_h = hu;
                    out_f = f;
                    if (bout && k == T - 1) {
                        bout[bidx(jl, 0)] = out_h;
                        bout[bidx(jl, 1)] = out_f;
                    }
                }
                diag_in = up_h;
            }
            slab_off += (int64_t)max(width, 0) * T;
            prev_lo = lo;
            prev_hi = hi;
            __syncwarp();
        }

        // walk back from the end cell (the group's first lane)
        if (on && k == 0 && p >= 0) {
            const int64_t off = P.cig_off[p];
            const int64_t cap = P.cig_off[p + 1] - off;
            if (q.score <= 0) {
                P.cig_n[p] = 0;
            } else {
                RevCigar rcg{P.cig_ops + off, cap, 0, 0u, 0, false};
                rcg.push(4u, q.m - 1 - q.ie);  // trailing soft clip
                int32_t i = q.ie, jj = q.W - 1;
                int state = 0;
                // every step moves, or switches into a gap state before moving
                const int64_t limit = 2 * ((int64_t)q.rows + q.W) + 4;
                // words of chunk cc start after the windows of chunks 0..cc-1
                int cc = i / rc, clo, chi;
                int64_t cbase = 0;
                for (int c2 = 0; c2 < cc; ++c2) {
                    int l2, h2;
                    chunk_window(q, c2, rc, l2, h2);
                    cbase += (int64_t)max(h2 - l2 + 1, 0) * T;
                }
                chunk_window(q, cc, rc, clo, chi);
                bool ok = false;
                for (int64_t it = 0; it < limit; ++it) {
                    if (i < 0 || jj < 0) {
                        ok = state == 0;
                        break;
                    }
                    while (i < cc * rc) {  // moved up into the previous chunk
                        --cc;
                        chunk_window(q, cc, rc, clo, chi);
                        cbase -= (int64_t)max(chi - clo + 1, 0) * T;
                    }
                    if (jj < clo || jj > chi) break;  // left the band: inconsistent
                    const int kk = (i - cc * rc) / TB_ROWS, nib = i % TB_ROWS;
                    const int64_t widx = TILED ? ((int64_t)cc * WCAP + (jj - clo)) * 32 + lane
                                               : cbase + (int64_t)(jj - clo) * T + kk;
                    const uint32_t code = (slab[widx] >> (4 * nib)) & 0xFu;
                    if (state == 0) {
                        const uint32_t src = code & 3u;
                        if (src == 0u) {
                            ok = true;
                            break;
                        }
                        if (src == 1u) {
                            rcg.push(0u, 1);
                            --i;
                            --jj;
                        } else {
                            state = src == 2u ? 1 : 2;
                        }
                    } else if (state == 1) {
                        rcg.push(2u, 1);
                        if (code & 4u) state = 0;
                        --jj;
                    } else {
                        rcg.push(1u, 1);
                        if (code & 8u) state = 0;
                        --i;
                    }
                }
                if (!ok) atomicOr(L.status, ST_INTERNAL);
                rcg.push(4u, i + 1);  // leading soft clip
                rcg.flush();
                if (rcg.overflow) {
                    P.cig_n[p] = -1;
                    atomicOr(L.status, ST_CAPACITY);
                } else {
                    uint32_t *o = P.cig_ops + off;
                    for (int32_t a2 = 0, b2 = rcg.n - 1; a2 < b2; ++a2, --b2) {
                        const uint32_t tmp = o[a2];
                        o[a2] = o[b2];
                        o[b2] = tmp;
                    }
                    P.cig_n[p] = rcg.n;
                }
            }
        }
        __syncwarp();
    }
    }  // parts
}

// ---------------------------------------------------------------------------
// 16x2 traceback, one block of rows at a time.  It serves the classes whose
// score bound keeps every value below 32768 (match x min(m, n) <= 32000,
// match - o <= 127).  A group of T lanes owns two pairs, A in the low and B
// in the high half of every register, so each DPX instruction recomputes two
// cells.
//
// Blocks.  The score pass kept H and F of every column for the rows that end
// a block of 50 to 64 read rows (the checkpoints).  A pair's path is at
// (i, j) with the exact value v of its state; the block of row i is swept
// from the checkpoint above it (row i0 - 1, or the matrix edge) down to row
// i over the columns the path can use, the walk goes back through the block
// until it crosses row i0 or ends, and the next block starts from there.
//
// The columns.  A path that enters the block below checkpoint column j' with
// value h gains at most match per row, and its d = j - j' - (i - i0 + 1)
// deletions cost at least -o - (d - 1) e, so it can reach v only if
//   h + match (i - i0 + 1) + o + (d - 1) e >= v.
// D is the largest such d over the checkpoint's columns (and over paths that
// start inside the block, h = 0); the insertions are bounded likewise by the
// largest h.  Row r of the block then needs columns j - (i - r) - D ..
// j - (i - r) + I only: cells on optimal paths keep their exact values, all
// others can only come out lower, so every comparison of the walk comes out
// as in the full matrix.  From the path's side, the rows below r gain at most
// match each, so no more than (score - v + match (i - r) + o) / -e + 1
// deletions lie below row r, which narrows the last rows' windows.  The whole
// read's band is as wide as the loss of the whole read allows; a block's is
// as wide as its own loss.  Sweeping the 2M uneven pairs of 75 to 800 bases
// by whole-read bands took 45 ms, plus 7.5 ms for walks in kernels of their
// own.
//
// Sweep.  Lane k of a group holds 8 rows (4 with 16 lanes) of a chunk of 8T
// (64) rows on a one-step wavefront.  A lane stores two 32-bit words per
// window offset (rows 0-3 and rows 4-7; pair A in bits 0-15, pair B in bits
// 16-31), and its words of four consecutive offsets share one 32-byte sector:
// uint2
// [((chunk x S4 + t / 4) x 32 + lane) x 4 + t % 4].  Per cell four bits record
// which equalities fail (1 = not equal):
//   bit 0  H != H(i-1,j-1) + s    bit 1  H != E
//   bit 2  E != H(i,j-1) + o      bit 3  F != H(i-1,j) + o
// Each bit is min(x, 1) per half of a difference x that is non-negative in
// both halves (a maximum minus one of its operands), so the differences and
// the packing of the bits are integer multiply-adds on the FMA pipe, next to
// the DPX maxima on the ALU pipe: per two cells 9 ALU and 9 FMA-pipe
// instructions when s - o >= 0 for every substitution (FMA_ADD), else the
// diagonal add and its difference move to the ALU pipe.
//
// Each pair keeps its own chunk windows; both pairs of a lane step through
// window offset t together and the warp steps to its widest window.  Offsets
// past a pair's own window are computed as well: they lie right of its box
// and hold values no larger than the full matrix's (past the window end they
// see an all-(s = o) table, so nothing grows there), which changes no cell
// the walk reads.  Boundary rows between chunks hold (H | F << 16) per pair
// and offset and are updated in place; the block's checkpoint columns are
// copied into the same row first.  Windows start at multiples of four
// columns, so a boundary row is read four offsets at a time, one group of
// four steps before it is used: a step takes the SM's 16 warps about 560
// cycles to issue, an L2 load under this traffic longer.  The rows (and the
// tiles) bypass the L1, which they would overflow; reads, windows and
// checkpoints then stay in it.
//
// Walk.  The path takes the diagonal where bit 0 is clear, else E where bit 1
// is clear, else F, and a gap run opens where bit 2 (3) is clear.  Whether H
// is 0 is not stored: the walk carries the exact value of its state, starting
// from the score, and stops where H reaches 0.  Where the read and window
// bases are equal the diagonal always holds (H(i,j) <= H(i-1,j-1) + match:
// dropping the last aligned pair of an alignment that ends at (i,j) leaves
// one that reaches (i-1,j-1) with the same gap), so the walk skips runs of
// equal bases 16 at a time and reads the tile at mismatches and gaps only.
// A lane with two pairs to walk (T = 1) takes a step of each per iteration,
// their loads in flight together.

__device__ __forceinline__ uint32_t mad_u32(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

__device__ __forceinline__ uint32_t min_u16x2(uint32_t a, uint32_t b)
{
    uint32_t d;
    asm("min.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

__device__ __forceinline__ uint32_t splat16(int32_t x) { return ((uint32_t)(uint16_t)(int16_t)x) * 0x10001u; }

// Selector nibbles of one row for pair A (bytes 0-1) and pair B (bytes 2-3):
// the row's base picks its byte of the column table and the high byte
// replicates its sign; a row without a base takes the sign of byte 0 (0 or
// -1, never above s = o).
__device__ __forceinline__ uint32_t sel16(uint32_t xa, uint32_t xb)
{
    const uint32_t a = xa < 4u ? (xa | ((8u | xa) << 4)) : 0x88u;
    const uint32_t b = xb < 4u ? ((4u + xb) | ((12u + xb) << 4)) : 0xCCu;
    return a | (b << 8);
}

// Bases pos - 15 .. pos of a packed buffer, base pos in the top two bits
// (before the buffer's start: zeros).
__device__ __forceinline__ uint32_t bases_back(const uint32_t *__restrict__ buf, int64_t pos)
{
    const int64_t w = pos >> 4;
    const uint32_t hi = __ldg(buf + w);
    const uint32_t lo = ((pos & 15) != 15 && w > 0) ? __ldg(buf + w - 1) : 0u;
    return __funnelshift_rc(lo, hi, 2 * (int)(pos & 15) + 2);
}

// The pairs of a warp's task, one entry per pair: path position (i, j), the
// exact value v of its state st (0 H, 1 E, 2 F, -1 no more to do), the
// current block's first row i0 and band limits D and I, and the CIGAR so far
// (cn runs written below the slot's end out, then a run of len x op).
template <int PAIRS>
struct TaskPairs {
    int64_t rs[PAIRS], ws[PAIRS], out[PAIRS];
    uint32_t ck[PAIRS];
    int32_t ck_row[PAIRS];
    int32_t p[PAIRS], n[PAIRS], S[PAIRS], cap[PAIRS];
    int32_t i[PAIRS], j[PAIRS], v[PAIRS], st[PAIRS];
    int32_t i0[PAIRS], D[PAIRS], I[PAIRS];
    int32_t cn[PAIRS], op[PAIRS], len[PAIRS];
};

// num / d for d >= 1 (the common gap extension of 1 needs no division).
__device__ __forceinline__ int32_t div_by(int32_t num, int32_t d) { return d == 1 ? num : num / d; }

// Most deletions an alignment part can hold that may lose `num` more than
// the opening of one gap (num < 0: none); -ge = nge = 0: no limit.
__device__ __forceinline__ int32_t max_del(int32_t num, int32_t nge)
{
    if (nge == 0) return 1 << 24;
    return num < 0 ? 0 : div_by(num, nge) + 1;
}

// First window column (a multiple of 4) of the rows from r0 on of a block
// entered at (i, j) with value v: D deletions at most, and no more than the
// rows below r0 can pay for.
__device__ __forceinline__ int32_t block_lo(int32_t i, int32_t j, int32_t v, int32_t D, int32_t S, int32_t r0,
                                            const Scoring &sc)
{
    const int32_t back = i - r0;
    const int32_t d = min(D, max_del(S - v + sc.ma * back + sc.go, -sc.ge));
    return max(0, j - back - d) & ~3;
}

__device__ __forceinline__ uint32_t quad_at(const uint4 &q, int s)
{
    return s == 0 ? q.x : s == 1 ? q.y : s == 2 ? q.z : q.w;
}

template <int T, bool FMA_ADD>
__global__ void __launch_bounds__(128, 4) k_traceback16(const TracebackLaunch L)
{
    constexpr int G = 32 / T;       // groups per warp, two pairs each
    constexpr int PAIRS = 2 * G;    // pairs per task
    constexpr int ROWS = tb16_rows(T);  // rows per lane
    constexpr int rc = T * ROWS;        // rows per chunk
    const TbParams &P = L.P;
    // s_tab[w] byte x = s(x, w) - o; s_tab[4] = 0 (s = o, past a window end)
    __shared__ uint32_t s_tab[8];
    {
        const uint32_t mis4 = ((uint32_t)(uint8_t)(int8_t)(P.sc.mi - P.sc.go)) * 0x01010101u;
        const uint32_t ma4 = ((uint32_t)(uint8_t)(int8_t)(P.sc.ma - P.sc.go)) * 0x01010101u;
        if (threadIdx.x < 4) s_tab[threadIdx.x] = prmt(mis4, ma4, 0x3210u + (4u << (4u * threadIdx.x)));
        else if (threadIdx.x < 8) s_tab[threadIdx.x] = 0u;
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int g = lane / T, k = lane % T;
    const int64_t warp_global = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const DevTbPlan &dp = *L.dp;
    // input already found invalid (an unsupported size means some pairs were
    // not scored, so the traceback order is incomplete): do nothing
    if (*(volatile const int32_t *)L.status & (ST_BAD_INPUT | ST_UNSUPPORTED)) return;
    // (the variants of one launch share the size of a slot)
    uint32_t *const slot = L.slab + dp.var_slot_offset[L.variant] + warp_global * dp.var_slot_words[L.variant];
    const uint32_t GE2 = splat16(P.sc.ge), GO2 = splat16(P.sc.go);
    const uint32_t one = (uint32_t)L.one;
    const uint32_t m1 = 0u - one, two = one + one, four = two + two, eight = four + four;
    const uint32_t mul1 = eight + eight, mul2 = mul1 * mul1, mul3 = mul2 * mul1;  // 16, 256, 4096
    const uint32_t ONES = 0x00010001u;

    __shared__ TaskPairs<PAIRS> s_task[4];  // 128 threads: 4 warps
    TaskPairs<PAIRS> &tp = s_task[threadIdx.x >> 5];
    // The part's values live in shared memory, one record per warp, read
    // where they are used (held in registers across the sweep they would
    // crowd out the sweep's own).
    struct PartCtx {
        const int32_t *order;
        int32_t *ctr;
        uint4 *bnd;
        int64_t lane_chunks;
        int32_t n_items, wcap, s4, block_rows, pi;
    };
    __shared__ PartCtx s_pc[4];
    volatile PartCtx *const pc = &s_pc[threadIdx.x >> 5];
    for (int v = L.variant; v < L.variant + L.n_variants; ++v) {
    if (warp_global >= dp.var_warps[v]) continue;  // no scratch slot
    __syncwarp();
    if (lane == 0) pc->pi = 0;
    __syncwarp();
    for (; pc->pi < dp.var_n[v]; next_index(pc->pi, lane)) {
    if (lane == 0) {
        const TbPartPlan &pp = dp.part[dp.var_part[v][pc->pi]];
        const int32_t s4 = (pp.wcap + T - 1 + 3) >> 2;
        pc->order = L.order + pp.start;
        pc->ctr = L.work_counter + kTbParts * pp.cls + pp.part;
        pc->bnd = (uint4 *)(slot + ((32 * pp.slab_words + 63) & ~(int64_t)63));
        pc->lane_chunks = pp.slab_words / (ROWS * (int64_t)max(s4, 1));
        pc->n_items = pp.count;
        pc->wcap = pp.wcap;
        pc->s4 = s4;
        pc->block_rows = pp.block_rows;
    }
    __syncwarp();

    for (;;) {
        int base = 0;
        if (lane == 0) base = atomicAdd(pc->ctr, PAIRS);
        base = __shfl_sync(FULLMASK, base, 0);
        if (base >= pc->n_items) break;
        for (int wi = lane; wi < PAIRS; wi += 32) {
            const int32_t p = base + wi < pc->n_items ? pc->order[base + wi] : -1;
            const TbPair q = tb_pair(P, p, L.status);
            tp.p[wi] = p;
            tp.rs[wi] = q.rs;
            tp.ws[wi] = q.ws;
            tp.n[wi] = q.n;
            tp.S[wi] = tp.v[wi] = q.score;
            tp.i[wi] = q.ie;
            tp.j[wi] = q.je;
            tp.st[wi] = q.score > 0 ? 0 : -1;
            tp.cn[wi] = 0;
            tp.op[wi] = 4;  // trailing soft clip
            tp.len[wi] = q.m - 1 - q.ie;
            tp.ck[wi] = 0;
            tp.ck_row[wi] = 0;
            const int64_t o0 = p >= 0 ? P.cig_off[p] : 0, o1 = p >= 0 ? P.cig_off[p + 1] : 0;
            tp.out[wi] = o1;
            tp.cap[wi] = (int32_t)lmin(o1 - o0, INT32_MAX);
            if (p >= 0 && q.score <= 0) P.cig_n[p] = 0;
            if (q.score > 0 && pc->block_rows) {
                const uint2 c = P.ck_pos[p];
                tp.ck[wi] = c.x;
                tp.ck_row[wi] = (int32_t)c.y;
            }
        }
        __syncwarp();

        for (;;) {
            // the next block of every pair that is not done: its first row
            // and band limits
            bool any = false, any_top = false;
            int rows_l = 0;
#pragma unroll 1
            for (int x = 0; x < 2; ++x) {
                const int wi = 2 * g + x;
                const bool act = tp.st[wi] >= 0;
                const int32_t i = tp.i[wi], j = tp.j[wi], vv = tp.v[wi], S = tp.S[wi];
                const int32_t br = pc->block_rows, ma = P.sc.ma, go = P.sc.go, nge = -P.sc.ge;
                const int32_t blk = act && br ? i / br : 0;
                const int32_t i0 = blk * br;
                const int32_t nrow = act ? i - i0 + 1 : 0;
                const int32_t gain = ma * nrow - vv;
                int32_t D = max_del(gain + go, nge), M = 0;
                if (act && i0 > 0) {
                    const int32_t dcap = max_del(gain + go + min(S, ma * i0), nge);
                    const int32_t jmin = max(0, j - nrow - dcap);
                    const uint4 *row = P.ck_pool + tp.ck[wi] + (int64_t)(blk - 1) * (tp.ck_row[wi] >> 1);
                    const int sh = 16 * (tp.ck_row[wi] & 1);
#pragma unroll 4
                    for (int u = (j >> 1) - k; u >= (jmin >> 1); u -= T) {
                        const uint4 q = __ldg(row + u);
                        const int32_t h0 = (int32_t)((q.x >> sh) & 0xFFFFu), h1 = (int32_t)((q.z >> sh) & 0xFFFFu);
                        M = max(M, max(h0, h1));
                        const int32_t d = j - 2 * u - nrow;
                        if (d >= 1 && (d - 1) * nge <= gain + go + h0) D = max(D, d);
                        if (d >= 2 && (d - 2) * nge <= gain + go + h1) D = max(D, d - 1);
                    }
                }
#pragma unroll
                for (int o = 1; o < T; o <<= 1) {
                    D = max(D, __shfl_xor_sync(FULLMASK, D, o));
                    M = max(M, __shfl_xor_sync(FULLMASK, M, o));
                }
                const int32_t inum = i0 > 0 ? gain + M : gain + go + nge;
                __syncwarp();
                if (act && k == 0) {
                    tp.i0[wi] = i0;
                    tp.D[wi] = D;
                    tp.I[wi] = inum < 0 ? 0 : inum / (ma + nge);
                    if ((nrow + rc - 1) / rc > pc->lane_chunks) {  // never overrun the tile
                        atomicOr(L.status, ST_INTERNAL);
                        P.cig_n[tp.p[wi]] = 0;
                        tp.st[wi] = -1;
                    }
                }
                __syncwarp();
                if (tp.st[wi] >= 0) {
                    any = true;
                    any_top |= i0 > 0;
                    rows_l = max(rows_l, nrow);
                }
            }
            if (!__any_sync(FULLMASK, any)) break;
            any_top = __any_sync(FULLMASK, any_top);
            const int chunks = ((int)__reduce_max_sync(FULLMASK, (unsigned)rows_l) + rc - 1) / rc;

            int prev_lo[2] = {0, 0};
            int prev_groups = 0;  // groups of four offsets of the boundary row that hold values
            for (int c = 0; c < chunks; ++c) {
                int lo[2], hi[2], rem[2];
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int wi = 2 * g + x;
                    lo[x] = 0;
                    hi[x] = -1;
                    rem[x] = 0;
                    const int32_t i = tp.i[wi], j = tp.j[wi], r0 = tp.i0[wi] + c * rc;
                    if (tp.st[wi] >= 0 && r0 <= i) {
                        lo[x] = block_lo(i, j, tp.v[wi], tp.D[wi], tp.S[wi], r0, P.sc);
                        hi[x] = min(j, j - (i - min(r0 + rc - 1, i)) + tp.I[wi]);
                        if (hi[x] - lo[x] >= pc->wcap) {  // never overrun the tile or the boundary row
                            if (k == 0) atomicOr(L.status, ST_INTERNAL);
                            hi[x] = lo[x] + pc->wcap - 1;
                        }
                        rem[x] = tp.n[wi] - lo[x];  // window columns from lo on
                    }
                }
                // offsets, in groups of four
                const int groups =
                    ((int)__reduce_max_sync(FULLMASK, (unsigned)max(max(hi[0] - lo[0] + 1, hi[1] - lo[1] + 1), 0)) +
                     3) >> 2;
                const int steps = 4 * groups + T - 1;
                uint4 *const bnd = pc->bnd + 2 * g;  // group q of pair x at bnd[2 * G * q + x]
                if (c == 0 && any_top) {
                    // the checkpoint's columns from lo - 4 on, as a boundary
                    // row (zeros for a pair whose block starts at row 0)
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const int wi = 2 * g + x;
                        const bool top = hi[x] >= lo[x] && tp.i0[wi] > 0;
                        const int32_t n = tp.n[wi];
                        const int sh = 16 * (tp.ck_row[wi] & 1);
                        const uint4 *row = P.ck_pool + tp.ck[wi] +
                                           (int64_t)(top ? tp.i0[wi] / pc->block_rows - 1 : 0) * (tp.ck_row[wi] >> 1);
                        auto hf = [&](uint32_t h, uint32_t f) { return ((h >> sh) & 0xFFFFu) | ((f >> sh) << 16); };
                        prev_lo[x] = lo[x] - 4;
#pragma unroll 4
                        for (int q = k; q <= groups; q += T) {
                            const int col = lo[x] - 4 + 4 * q;
                            uint4 w = make_uint4(0u, 0u, 0u, 0u);
                            if (top && col >= 0 && col < n) {
                                const uint4 a = __ldg(row + (col >> 1));
                                const uint4 b = col + 2 < n ? __ldg(row + (col >> 1) + 1) : w;
                                w.x = hf(a.x, a.y);
                                if (col + 1 < n) w.y = hf(a.z, a.w);
                                w.z = hf(b.x, b.y);
                                if (col + 3 < n) w.w = hf(b.z, b.w);
                            }
                            __stcg(bnd + 2 * G * q + x, w);
                        }
                    }
                    prev_groups = groups + 1;
                    __syncwarp();
                }
                // one boundary row, updated in place: the first lane reads
                // group q + shift (shift >= 0, in groups) before the last
                // lane overwrites group q; a pair without rows in this chunk
                // reads it at shift 0 (its values are never used)
                const bool has_in = (c > 0 || any_top) && k == 0;
                const bool has_out = c + 1 < chunks && k == T - 1;
                int shift[2];
#pragma unroll
                for (int x = 0; x < 2; ++x) shift[x] = hi[x] >= lo[x] ? max(lo[x] - prev_lo[x], 0) >> 2 : 0;
                auto bload = [&](int x, int q) -> uint4 {
                    return has_in && q >= 0 && q < prev_groups ? __ldcg(bnd + 2 * G * q + x)
                                                               : make_uint4(0u, 0u, 0u, 0u);
                };
                // the row above: packed (H | F << 16) of four offsets per pair
                const uint32_t dg0 = bload(0, shift[0] - 1).w, dg1 = bload(1, shift[1] - 1).w;
                uint4 nb[2] = {bload(0, shift[0]), bload(1, shift[1])};
                // the windows' first bases and the rows' (while those loads
                // are in flight)
                uint32_t codes[2], ww[2], wn[2];
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int wi = 2 * g + x;
                    ww[x] = 0u;
                    wn[x] = k == 0 && rem[x] > 0 ? load_bases(P.ps.wins, tp.ws[wi] + lo[x], min(16, rem[x])) : 0u;
                    codes[x] = 0x44444444u;  // 4 bits per row, 4 = no base
                    const int row = tp.i0[wi] + c * rc + k * ROWS;
                    const int cnt = rem[x] > 0 ? min(ROWS, tp.i[wi] - row + 1) : 0;
                    if (cnt > 0) {
                        const uint32_t w = load_bases(P.ps.reads, tp.rs[wi] + row, cnt);
#pragma unroll
                        for (int r = 0; r < ROWS; ++r)
                            if (r < cnt)
                                codes[x] = (codes[x] & ~(0xFu << (4 * r))) | (((w >> (2 * r)) & 3u) << (4 * r));
                    }
                }
                uint32_t sel[ROWS];
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
                    sel[r] = sel16((codes[0] >> (4 * r)) & 0xFu, (codes[1] >> (4 * r)) & 0xFu);
                uint32_t E[ROWS], Hp[ROWS];
#pragma unroll
                for (int r = 0; r < ROWS; ++r) {
                    E[r] = 0u;
                    Hp[r] = 0u;
                }
                uint32_t diag_in = prmt(dg0, dg1, 0x5410u);
                uint32_t out_h = 0u, out_f = 0u, bases = 0u;
                // a lane's words of four steps: 32 bytes (16 with four rows)
                uint4 *tile = (uint4 *)slot + ((int64_t)c * pc->s4 * 32 + lane) * (ROWS / 4);

                for (int t0 = 0; t0 < steps; t0 += 4) {
                    uint4 nx[2], ob[2];
#pragma unroll
                    for (int x = 0; x < 2; ++x) nx[x] = bload(x, shift[x] + (t0 >> 2) + 1);
#pragma unroll 1
                    for (int half = 0; half < 2; ++half) {
                    uint4 wq;
#pragma unroll
                    for (int s = 0; s < 2; ++s) {
                        const int t = t0 + 2 * half + s;
                        // the row above: from the lane before (its last
                        // step), or the boundary row for the group's first
                        // lane
                        uint32_t up_h = T > 1 ? __shfl_up_sync(FULLMASK, out_h, 1) : 0u;
                        uint32_t up_f = T > 1 ? __shfl_up_sync(FULLMASK, out_f, 1) : 0u;
                        if (k == 0) {
                            const uint32_t a = quad_at(nb[0], s), b = quad_at(nb[1], s);
                            up_h = prmt(a, b, 0x5410u);
                            up_f = prmt(a, b, 0x7632u);
                        }
                        const int jl = t - k;  // this lane's window offset
                        uint32_t w0 = 0u, w1 = 0u;
                        // the column's bases (4: past the window) of both
                        // pairs: the first lane streams them, 16 columns
                        // requested 16 columns ahead, and each lane takes
                        // the lane before's of the last step (with a stream
                        // per lane some lane refilled its own at every step)
                        if (s == 0 && (t & 15) == 0 && k == 0) {
#pragma unroll
                            for (int x = 0; x < 2; ++x) {
                                ww[x] = wn[x];
                                const int left = rem[x] - t - 16;
                                wn[x] = left > 0 ? load_bases(P.ps.wins, tp.ws[2 * g + x] + lo[x] + t + 16,
                                                              min(16, left))
                                                 : 0u;
                            }
                        }
                        const uint32_t bprev = T > 1 ? __shfl_up_sync(FULLMASK, bases, 1) : 0u;
                        bases = (t < rem[0] ? ww[0] & 3u : 4u) | ((t < rem[1] ? ww[1] & 3u : 4u) << 3);
                        ww[0] >>= 2;
                        ww[1] >>= 2;
                        if (T > 1 && k > 0) bases = bprev;
                        if (T == 1 || jl >= 0) {
                            const uint32_t tA = s_tab[bases & 7u], tB = s_tab[bases >> 3];
                            uint32_t d0 = diag_in, hu = up_h, f = up_f;
#pragma unroll
                            for (int r = 0; r < ROWS; ++r) {
                                const uint32_t sp = prmt(tA, tB, sel[r]);  // s - o, both pairs
                                const uint32_t e = __viaddmax_s16x2(E[r], GE2, Hp[r]);
                                f = __viaddmax_s16x2(f, GE2, hu);
                                const uint32_t d =
                                    FMA_ADD ? mad_u32(d0, one, sp) : __viaddmax_s16x2(d0, sp, 0x80008000u);
                                const uint32_t u = __vimax3_s16x2(d, e, f);
                                const uint32_t h = __viaddmax_s16x2_relu(u, GO2, 0u);
                                const uint32_t nd =
                                    FMA_ADD ? min_u16x2(mad_u32(d, m1, u), ONES) : min_u16x2(u ^ d, ONES);
                                const uint32_t ne = min_u16x2(mad_u32(e, m1, u), ONES);
                                const uint32_t nE = min_u16x2(mad_u32(Hp[r], m1, e), ONES);
                                const uint32_t nF = min_u16x2(mad_u32(hu, m1, f), ONES);
                                uint32_t code = mad_u32(ne, two, nd);
                                code = mad_u32(nE, four, code);
                                code = mad_u32(nF, eight, code);
                                if (r == 0) w0 = code;
                                else if (r == 4) w1 = code;
                                else if (r < 4) w0 = mad_u32(code, r == 1 ? mul1 : r == 2 ? mul2 : mul3, w0);
                                else w1 = mad_u32(code, r == 5 ? mul1 : r == 6 ? mul2 : mul3, w1);
                                d0 = Hp[r];
                                Hp[r] = h;
                                E[r] = e;
                                hu = h;
                            }
                            out_h = hu;
                            out_f = f;
                            diag_in = up_h;
                            const uint32_t o0 = prmt(hu, f, 0x5410u), o1 = prmt(hu, f, 0x7632u);
                            if (T == 1) {
                                (s == 0 ? ob[0].z : ob[0].w) = o0;
                                (s == 0 ? ob[1].z : ob[1].w) = o1;
                            } else if (has_out) {
                                uint32_t *const w = (uint32_t *)(bnd + 2 * G * (jl >> 2)) + (jl & 3);
                                __stcg(w, o0);
                                __stcg(w + 4, o1);
                            }
                        }
                        (s == 0 ? wq.x : wq.z) = w0;
                        (s == 0 ? wq.y : wq.w) = w1;
                    }
                    if (ROWS == 8) __stcg(tile + half, wq);
                    else __stcg((uint2 *)tile + half, make_uint2(wq.x, wq.z));
                    if (half == 0) {
#pragma unroll
                        for (int x = 0; x < 2; ++x) {
                            nb[x].x = nb[x].z;
                            nb[x].y = nb[x].w;
                            ob[x].x = ob[x].z;
                            ob[x].y = ob[x].w;
                        }
                    }
                    }
                    tile += 32 * (ROWS / 4);
                    if (T == 1 && has_out) {
                        __stcg(bnd + 2 * G * (t0 >> 2), ob[0]);
                        __stcg(bnd + 2 * G * (t0 >> 2) + 1, ob[1]);
                    }
                    nb[0] = nx[0];
                    nb[1] = nx[1];
                }
                prev_lo[0] = lo[0];
                prev_lo[1] = lo[1];
                prev_groups = groups;
                __syncwarp();
            }

            // the walks back through the block: lanes 0 and 1 of a group one
            // pair each, or with T = 1 a lane both of its pairs
            constexpr int NW = T == 1 ? 2 : 1;
            int wst_[NW], wi_[NW], i_[NW], j_[NW], v_[NW], cn_[NW], len_[NW], cl_[NW], lo_[NW];
            uint32_t op_[NW];
            bool go_[NW], fin_[NW], ok_[NW];
            bool more = false;
#pragma unroll
            for (int x = 0; x < NW; ++x) {
                const int wi = 2 * g + (T == 1 ? x : min(k, 1));
                wi_[x] = wi;
                wst_[x] = tp.st[wi];
                i_[x] = tp.i[wi];
                j_[x] = tp.j[wi];
                v_[x] = tp.v[wi];
                cn_[x] = tp.cn[wi];
                len_[x] = tp.len[wi];
                op_[x] = (uint32_t)tp.op[wi];
                cl_[x] = -1;
                lo_[x] = 0;
                go_[x] = (T == 1 || k < 2) && wst_[x] >= 0;
                fin_[x] = false;
                ok_[x] = true;
                more |= go_[x];
            }
            const int S4 = pc->s4, wcap = pc->wcap;
            auto push = [&](int x, uint32_t o, int32_t l) {
                if (o == op_[x]) {
                    len_[x] += l;
                    return;
                }
                if (len_[x] > 0) {  // runs are parked downwards from the slot's end
                    if (cn_[x] < tp.cap[wi_[x]])
                        P.cig_ops[tp.out[wi_[x]] - 1 - cn_[x]] = ((uint32_t)len_[x] << 4) | op_[x];
                    ++cn_[x];
                }
                op_[x] = o;
                len_[x] = l;
            };
            // the walk's end, or its exit from the block
            auto stopped = [&](int x) {
                if (wst_[x] == 0 && v_[x] == 0) fin_[x] = true;
                else if (wst_[x] == 1 || i_[x] >= tp.i0[wi_[x]]) {
                    if (j_[x] >= 0 && v_[x] >= 0) return false;
                    ok_[x] = false;
                }
                return true;
            };
#pragma unroll
            for (int x = 0; x < NW; ++x)
                if (go_[x] && stopped(x)) go_[x] = false;
            while (more) {
                // equal bases: the diagonal
                uint32_t diff[NW];
#pragma unroll
                for (int x = 0; x < NW; ++x) {
                    const bool need = go_[x] && wst_[x] == 0;
                    const int64_t r = need ? tp.rs[wi_[x]] + i_[x] : 0, w = need ? tp.ws[wi_[x]] + j_[x] : 0;
                    diff[x] = bases_back(P.ps.reads, r) ^ bases_back(P.ps.wins, w);
                }
                bool cell[NW];  // a cell of the tile decides the next step
#pragma unroll
                for (int x = 0; x < NW; ++x) {
                    cell[x] = go_[x];
                    if (go_[x] && wst_[x] == 0) {
                        const int same = min(__clz((int)diff[x]) >> 1, 16);
                        const int run = min(same, min(i_[x] - tp.i0[wi_[x]], j_[x]) + 1);
                        if (run > 0) {
                            push(x, 0u, run);
                            i_[x] -= run;
                            j_[x] -= run;
                            v_[x] -= run * P.sc.ma;
                            if (stopped(x)) go_[x] = false;
                            cell[x] = go_[x] && same < 16;
                        }
                    }
                }
                uint2 word[NW];
                int row[NW], run_cols[NW];
                uint32_t run_bits[NW];
#pragma unroll
                for (int x = 0; x < NW; ++x) {
                    row[x] = run_cols[x] = 0;
                    run_bits[x] = 0u;
                    word[x] = make_uint2(0u, 0u);
                    if (cell[x]) {
                        const int wi = wi_[x];
                        const int rel = i_[x] - tp.i0[wi], c = rel / rc;
                        if (c != cl_[x]) {
                            cl_[x] = c;
                            lo_[x] = block_lo(tp.i[wi], tp.j[wi], tp.v[wi], tp.D[wi], tp.S[wi], tp.i0[wi] + c * rc,
                                              P.sc);
                        }
                        const int jl = j_[x] - lo_[x], kk = (rel - c * rc) / ROWS, t = jl + kk;
                        row[x] = rel % ROWS;
                        if (jl < 0 || jl >= wcap) {  // left the band: inconsistent
                            ok_[x] = go_[x] = cell[x] = false;
                        } else {
                            const int64_t sector = ((int64_t)c * S4 + (t >> 2)) * 32 + g * T + kk;
                            if (ROWS == 8) word[x] = __ldcg((const uint2 *)slot + 4 * sector + (t & 3));
                            else word[x].x = __ldcg(slot + 4 * sector + (t & 3));
                            // a deletion run under way: up to three columns
                            // more of this sector (an intron's run is
                            // hundreds of columns)
                            if (wst_[x] == 1 && (t & 3) > 0 && jl > 0) {
                                const int bit = 16 * (wi & 1) + 4 * (row[x] & 3) + 2;
                                run_cols[x] = min(t & 3, jl);
#pragma unroll
                                for (int q = 1; q < 4; ++q)
                                    if (q <= run_cols[x]) {
                                        const int64_t at = 4 * sector + (t & 3) - q;
                                        const uint32_t w = ROWS == 8
                                                               ? __ldcg(slot + 2 * at + (row[x] >> 2))
                                                               : __ldcg(slot + at);
                                        run_bits[x] |= ((w >> bit) & 1u) << q;
                                    }
                            }
                        }
                    }
                }
                more = false;
#pragma unroll
                for (int x = 0; x < NW; ++x) {
                    if (cell[x]) {
                        const uint32_t code =
                            ((row[x] < 4 ? word[x].x : word[x].y) >> (16 * (wi_[x] & 1) + 4 * (row[x] & 3))) & 0xFu;
                        if (wst_[x] == 0 && (code & 1u)) wst_[x] = (code & 2u) ? 2 : 1;
                        if (wst_[x] == 0) {
                            v_[x] -= P.sc.mi;  // H(i-1, j-1) = H(i, j) - s
                            push(x, 0u, 1);
                            --i_[x];
                            --j_[x];
                        } else {
                            // E(i,j) = H(i,j-1) + o or E(i,j-1) + e, and F
                            // the same way up
                            const bool del = wst_[x] == 1;
                            int32_t cols = 1;
                            bool open = !(code & (del ? 4u : 8u));
                            if (del && !open) {
                                // extended columns of the sector, then
                                // perhaps the opening one
                                const int more_cols = run_cols[x];
#pragma unroll
                                for (int q = 1; q < 4; ++q)
                                    if (q <= more_cols && !open) {
                                        ++cols;
                                        open = !((run_bits[x] >> q) & 1u);
                                    }
                            }
                            push(x, del ? 2u : 1u, cols);
                            v_[x] -= (cols - 1) * P.sc.ge + (open ? P.sc.go : P.sc.ge);
                            if (open) wst_[x] = 0;
                            if (del) j_[x] -= cols;
                            else --i_[x];
                        }
                        if (stopped(x)) go_[x] = false;
                    }
                    more |= go_[x];
                }
            }
#pragma unroll
            for (int x = 0; x < NW; ++x) {
                const int wi = wi_[x];
                if (tp.st[wi] < 0 || (T > 1 && k >= 2)) continue;
                if (!fin_[x] && (i_[x] < 0 || !ok_[x])) {  // no zero reached: inconsistent
                    atomicOr(L.status, ST_INTERNAL);
                    fin_[x] = true;
                }
                if (fin_[x]) {
                    push(x, 4u, i_[x] + 1);  // leading soft clip
                    push(x, 5u, 0);
                    const int32_t cn = cn_[x], cap = tp.cap[wi], p = tp.p[wi];
                    if (cn > cap) {
                        P.cig_n[p] = -1;
                        atomicOr(L.status, ST_CAPACITY);
                    } else {
                        // the runs stand in order at the slot's end: move them down
                        uint32_t *const to = P.cig_ops + P.cig_off[p];
                        const uint32_t *const from = P.cig_ops + tp.out[wi] - cn;
                        if (to != from)
                            for (int32_t q = 0; q < cn; ++q) to[q] = from[q];
                        P.cig_n[p] = cn;
                    }
                    wst_[x] = -1;
                }
                tp.st[wi] = wst_[x];
                tp.i[wi] = i_[x];
                tp.j[wi] = j_[x];
                tp.v[wi] = v_[x];
                tp.cn[wi] = cn_[x];
                tp.op[wi] = (int32_t)op_[x];
                tp.len[wi] = len_[x];
            }
            __syncwarp();
        }
    }
    }  // parts
    }  // variants
}

// A device-planned launch of traceback variant v: the 16-bit kernel with
// tb16_variant_lanes(v) lanes per two pairs for v < N_TB16_VARIANTS, else the
// int32 kernel, tiled or with T lanes per pair.  fma: every substitution
// score minus gap_open is >= 0, so the 16-bit diagonal add can run on the
// FMA pipe.
static const void *tb16_kernel(int lanes, bool fma)
{
    switch (lanes) {
    case 1: return fma ? (const void *)k_traceback16<1, true> : (const void *)k_traceback16<1, false>;
    case 2: return fma ? (const void *)k_traceback16<2, true> : (const void *)k_traceback16<2, false>;
    case 4: return fma ? (const void *)k_traceback16<4, true> : (const void *)k_traceback16<4, false>;
    case 8: return fma ? (const void *)k_traceback16<8, true> : (const void *)k_traceback16<8, false>;
    default: return fma ? (const void *)k_traceback16<16, true> : (const void *)k_traceback16<16, false>;
    }
}

static const void *tb_kernel(int v, bool fma)
{
    if (v >= 0 && v < N_TB16_VARIANTS) return tb16_kernel(tb16_variant_lanes(v), fma);
    if (v == TB_VAR_TILED) return (const void *)k_traceback<true>;
    if (v == TB_VAR_GROUPED) return (const void *)k_traceback<false>;
    return nullptr;
}

int launch_traceback_variant(int v, bool fma, const TracebackLaunch &L, int blocks, cudaStream_t st)
{
    const void *fn = tb_kernel(v, fma);
    if (!fn || !L.dp || blocks < 1) return SW_ERR_INTERNAL;
    TracebackLaunch V = L;
    V.variant = v;
    V.n_variants = tb_launch_variants(v);
    void *args[] = {&V};
    if (cuda_failed(cudaLaunchKernel(fn, dim3(blocks), dim3(128), args, 0, st))) return SW_ERR_CUDA;
    count_launch();
    return launch_status();
}

// Blocks of a full-occupancy launch of traceback variant v.
int traceback_variant_blocks(int v, int sm_count, int *blocks)
{
    const void *fn = tb_kernel(v, true);
    if (!fn) return SW_ERR_INTERNAL;
    int bps = 0;
    if (cuda_failed(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, 128, 0))) return SW_ERR_CUDA;
    *blocks = std::max(bps, 1) * sm_count;
    return SW_OK;
}

}  // namespace swgb
