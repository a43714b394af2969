// a8: Smith-Waterman of candidate pairs (Sec. IV-E, Sec. VI), three passes.
//
// Recurrences (a gap of length L costs open + (L-1)*extend):
//   E(i,j) = max(H(i,j-1) - o, E(i,j-1) - e)     F(i,j) = max(H(i-1,j) - o, F(i-1,j) - e)
//   H(i,j) = max(0, H(i-1,j-1) + s(q_i, t_j), F(i,j), E(i,j))
// Reported: the score S, the end = the first maximum in row-major order, and the
// alignment a traceback from the end selects when it prefers the diagonal, then F,
// then E, and a gap open over an extension (its begin, identities, columns).
//
// Pass 1 (the whole matrix, every pair): score and end only.  A group of 8, 16 or 32 lanes
//   takes two pairs that share the query (candidate lists are grouped by i; within a run
//   of pairs of one query they are taken in order of target length, so the matrices of a
//   warp match) and holds them in the two 16-bit halves of each register, so one 16x2
//   maximum or add advances both.  Lane l owns up to 32 consecutive query rows and at step
//   s computes column j = s - l, taking H/F of the row above from lane l-1
//   (__shfl_up_sync).  Scores come from a biased query profile in shared memory
//   (one byte per [target residue][query row]) shared by every warp of the CTA.  Each lane
//   keeps its best cell (H, row, column) and looks at a column only when it holds a value
//   that can replace the group's best, so the end is the row-major first maximum.
//   Pass 1 also stores, per pair of query rows, the largest H it met there.
//   Queries longer than one stripe of 32 * 32 rows go in stripes whose last row is
//   handed on through a per-warp buffer.
// Pass 2 (its own kernel, one warp per pair; a band around the path): an anchored DP
//   over the reversed prefixes from the end (ei, ej), row by row with up to 128 columns
//   per row (four per lane; antidiagonal by antidiagonal when a row needs more or the
//   gap costs have o < e).  A suffix of the traced path starting on row i scores S minus
//   the forward value before it, which is at most the largest H pass 1 met on row
//   i-1's pair of rows; cells below that threshold die, the path's suffixes all
//   survive, and the cells reaching S bound the begin.  Their extent gives a rectangle
//   that contains the whole traced path.
// Pass 3 (k_sw_band: inside the columns that pass 2 left each row, where it kept them;
//   k_sw_carry: the whole rectangle): the DP again with zero boundaries; each state
//   carries its begin cell and (identities << 16 | matched columns) along the predecessor a
//   traceback would take.  Inside a region holding the path, the path's cells keep
//   their values and every choice along it is the same, so the carry at the end cell
//   is the traceback's.  cols = span_q + span_t - matched.
// Pairs whose scores could reach SCORE_MAX (max score * shorter length), gap opens
// above GAP_MAX, and queries longer than the shared-memory profile take pass 3 over the
// whole matrix with the end tracked there instead (int32).
// Captured launch sequences (alignment plans) pass device-side counts: each kernel then
// reads its pair or segment count from device memory and does nothing when the input
// checks flagged the batch.
#include <algorithm>

#include "internal.cuh"

namespace {

constexpr int NEG = -1000000000;
constexpr int SW_THREADS = 256;
constexpr int SW_WARPS = SW_THREADS / 32;
constexpr int STRIPE1 = 512;               // profile bytes per residue come in whole multiples
constexpr int PAD_SCORE = -30000;
constexpr int SEG_MAX = 512;               // pairs per scheduling segment, at most

struct sw_score_out {                      // pass 1 result per pair
    int32_t score;
    int32_t end_i, end_j;
    int32_t rect_i, rect_j;                // pass 2: start of the bounding rectangle
    int32_t big;                           // 1: not scored by pass 1 (k_sw_carry takes the whole
                                           // matrix); 2: pass 2 listed the pair for k_sw_band
};

// The filter-only mode (PASTIS_SW_FILTERED): the traced path lies in the rectangle
// [rect_i, end_i] x [rect_j, end_j] (the whole up-left rectangle before pass 2 narrows
// it), so its span on the shorter sequence (i on equal lengths) is at most the
// rectangle's extent there.  An extent below the coverage bound means the pair cannot
// pass the filter, and its begin and carried statistics are never needed.
__device__ __forceinline__ bool cannot_cover(const sw_score_out &r, int lq, int lt, int cov) {
    const int ext = lq <= lt ? r.end_i + 1 - r.rect_i : r.end_j + 1 - r.rect_j;
    return 100 * ext < cov * min(lq, lt);
}

// ---------------------------------------------------------------------------------
// segments: runs of pairs with the same query, at most seg_len(pairs of the call) long
// ---------------------------------------------------------------------------------
// A power of two from 16 to SEG_MAX that leaves about 1,024 full segments, three or more for
// each resident CTA: longer segments share a profile and balance the warps of a CTA, shorter
// ones the CTAs.
__device__ __forceinline__ int seg_len(int64_t n) {
    int len = SEG_MAX;
    while (len > 16 && n < (int64_t)len * 1024) len >>= 1;
    return len;
}

// dn (captured launches): the pair count in device memory, n the capacity; 0 past it.
__global__ void k_seg_flags(const pastis_cand *pairs, int64_t n, uint32_t *flags, const int64_t *dn) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t m = dn ? *dn : n;
    flags[p] = p < m && (p == 0 || (p & (seg_len(m) - 1)) == 0 || pairs[p].i != pairs[p - 1].i) ? 1u : 0u;
}

// Segments run in order of query length, longest first (bins of 16 residues): the CTAs at
// work at one time then run the same few of pass 1's loop bodies (16 row counts for each of 8,
// 16 and 32 lanes, and for 32 lanes in stripes), which together exceed the instruction cache,
// and the last segments taken are the shortest.  Pass 1 in input order and so: 10^6 pairs of
// 20,000 proteins 49.0 and 44.1 ms, 10^5 of 1,000 residues 27.6 and 25.2 ms, of 5,000 proteins
// 56.9 and 54.6 ms.
constexpr int SEG_BINS = 128;
__device__ __forceinline__ int seg_bin(int64_t m) { return SEG_BINS - 1 - (int)min((int64_t)SEG_BINS - 1, m >> 4); }

// Also counts the segments of each length bin (hist, zeroed by the caller).
__global__ void k_seg_starts(const pastis_cand *pairs, const int64_t *qoffsets, const uint32_t *flags,
                             const uint32_t *off, int64_t n, int64_t *seg_start, uint32_t *hist, const int64_t *dn,
                             const int *chk) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const int64_t m = dn ? *dn : n;
    if (p < m && flags[p]) {
        seg_start[off[p]] = p;
        if (!(chk && (chk[0] | chk[1]))) {       // a refused batch's indexes are not to be followed
            const int i = pairs[p].i;
            atomicAdd(&hist[seg_bin(qoffsets[i + 1] - qoffsets[i])], 1u);
        }
    }
    if (p == m - 1) seg_start[off[p] + flags[p]] = m;
}

// order[] = the segments by length bin (any order within a bin); taken: one zeroed counter
// per bin.
__global__ void __launch_bounds__(256) k_seg_order(const pastis_cand *pairs, const int64_t *qoffsets,
                                                   const int64_t *seg_start, int64_t n_seg, const uint32_t *d_nseg,
                                                   const uint32_t *hist, uint32_t *taken, uint32_t *order,
                                                   const int *chk) {
    if (d_nseg) n_seg = *d_nseg;
    if (chk && (chk[0] | chk[1])) return;
    if ((int64_t)blockIdx.x * blockDim.x >= n_seg) return;
    __shared__ uint32_t s_base[SEG_BINS];
    if (threadIdx.x < SEG_BINS) {
        uint32_t b = 0;
        for (int x = 0; x < (int)threadIdx.x; ++x) b += hist[x];
        s_base[threadIdx.x] = b;
    }
    __syncthreads();
    const int64_t sg = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (sg >= n_seg) return;
    const int i = pairs[seg_start[sg]].i;
    const int b = seg_bin(qoffsets[i + 1] - qoffsets[i]);
    order[s_base[b] + atomicAdd(&taken[b], 1u)] = (uint32_t)sg;
}

// ---------------------------------------------------------------------------------
// pass 1: two pairs per warp, one in each 16-bit half of every register
// ---------------------------------------------------------------------------------
// Every state is a signed 16-bit half: H >= 0, E and F >= -o (a gap is at least as good
// as opening it from H >= 0), and nothing exceeds the best score plus one substitution,
// so with no score reaching SCORE_MAX all values fit.  Per-half adds wrap within their
// half, and the 16x2 maximum instructions (max(a + b, c) and max(a, b, c, 0)) advance
// both pairs at once.  The profile stores score + o in a signed byte, so o <= GAP_MAX.
constexpr int GAP_MAX = 64;
constexpr int SCORE_MAX = 32000;
constexpr uint32_t P2 = 0x00010001u;
constexpr int NRES = PASTIS_NSYM + 1;      // profile rows: the residues, then the pad residue
constexpr int PAD_RES = PASTIS_NSYM;       // stands for target columns past the shorter target

// prmt with the sign-replicate bit of its selector (bytes below 0x80 become 0x00)
__device__ __forceinline__ uint32_t prmt_sx(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
    return d;
}
// a * b + c as a multiply-add (b is the run-time 1 the kernel receives, so the add goes
// to the multiply-add pipe and leaves the integer ALU pipe to the maxima)
__device__ __forceinline__ uint32_t madd(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

struct end_cell { int h, i, j; };

// The profile holds one signed byte per (target residue, query row): score + o, and
// o - 64 (the lowest score) for the pad residue and past the query.  A group of G lanes
// holds G * LR query rows (a stripe), lane l the LR consecutive rows l * LR ..; per stripe
// the bytes lie in planes of 16 rows, lane l's rows 16 p .. 16 p + 15 at p * 16 G + 16 l, so
// a lane reads its rows of one column with one 16-byte load per plane and the lanes of a
// group read consecutive words.
constexpr int SLOT = 16;
constexpr int LR_MAX = 32;

// The layout of one query of m residues: G lanes a pair, LR (even) rows a lane, ns stripes.
// A column step costs a lane about 10 cycles of the integer pipe per row (five 16x2
// instructions at half rate) and STEP_ROWS rows' worth of work that does not depend on
// LR (shuffles, window, addresses, the test for a new best), and a sweep takes n + G - 1
// steps; so few lanes with many rows each cost least per cell, but leave more pairs to a
// grab.  The fewest cycles of the CTA's slowest warp over the cnt pairs of the segment,
// with nt the longest target, decide.  More than one stripe takes 32 lanes.  `extra` (the
// layout the tuner picked for the query's length bin): 32 lanes and that many stripes more
// than needed, which pad fewer rows but sweep the target more often.  A query whose
// profile would not fit prow_cap bytes per residue so takes stripes of 512 rows, the densest
// profile.  The layout changes no result.
constexpr int STEP_ROWS = 3;
struct sw_tile { int G, lr, ns, prow; };

__device__ __forceinline__ sw_tile make_tile(int m, int G, int ns) {
    sw_tile t;
    const int per = (m + G * ns - 1) / (G * ns);
    t.G = G;
    t.ns = ns;
    t.lr = min(LR_MAX, max(2, (per + 1) & ~1));
    t.prow = ns * G * (t.lr > SLOT ? 2 * SLOT : SLOT);
    return t;
}

__device__ sw_tile pick_tile(int m, int extra, int cnt, int nt, int prow_cap) {
    const int need = max(1, (m + 32 * LR_MAX - 1) / (32 * LR_MAX));
    sw_tile best = make_tile(m, 32, need + extra);
    if (extra == 0 && need == 1) {
        int cost = 0x7FFFFFFF;
        for (int G = 32; G >= 8 && m <= G * LR_MAX; G >>= 1) {
            const sw_tile t = make_tile(m, G, 1);
            const int grabs = (cnt * G + 63) / 64;                  // of 64 / G pairs
            const int c = ((grabs + SW_WARPS - 1) / SW_WARPS) * (nt + G) * (t.lr + STEP_ROWS);
            if (c < cost) { cost = c; best = t; }
        }
    }
    if (best.prow > prow_cap) {
        best.G = 32;
        best.lr = SLOT;
        best.ns = max(1, (m + 511) / 512);
        best.prow = best.ns * 512;
    }
    return best;
}

// One column of a lane's LR rows for both pairs.  Ho = H - o is kept per row (it feeds
// E, F and the maxima), so the diagonal term is Ho(i-1, j-1) + (score + o).  rm keeps the
// largest Ho of each pair of rows over the columns (pass 2's bound); cm returns the
// largest Ho of this column, and tm where no row exceeds it.
template <int LR, int PLANE>
__device__ __forceinline__ uint32_t column2(const uint8_t *__restrict__ pa, const uint8_t *__restrict__ pb,
                                            uint32_t (&Ho)[LR], uint32_t (&E)[LR], uint32_t (&rm)[LR / 2],
                                            uint32_t hdiag, uint32_t &f, uint32_t &hup, uint32_t tm, uint32_t OP,
                                            uint32_t nEP) {
    // byte r of the two words into the low and high halves, sign-extended
    constexpr uint32_t SEL[4] = {0xc480u, 0xd591u, 0xe6a2u, 0xf7b3u};
    constexpr int PLANES = (LR + SLOT - 1) / SLOT;
    uint32_t wa[4 * PLANES], wb[4 * PLANES];
#pragma unroll
    for (int p = 0; p < PLANES; ++p) {
        const uint4 x = *reinterpret_cast<const uint4 *>(pa + p * PLANE);
        const uint4 y = *reinterpret_cast<const uint4 *>(pb + p * PLANE);
        wa[4 * p] = x.x; wa[4 * p + 1] = x.y; wa[4 * p + 2] = x.z; wa[4 * p + 3] = x.w;
        wb[4 * p] = y.x; wb[4 * p + 1] = y.y; wb[4 * p + 2] = y.z; wb[4 * p + 3] = y.w;
    }
    uint32_t cm = tm;
    uint32_t d = __vadd2(hdiag, prmt_sx(wa[0], wb[0], SEL[0]));   // H(i-1, j-1) + score
#pragma unroll
    for (int r = 0; r < LR; ++r) {
        // the next row's diagonal term is formed before this row's Ho is replaced, so each
        // row keeps its register from column to column
        uint32_t dn = 0u;
        if (r + 1 < LR) dn = __vadd2(Ho[r], prmt_sx(wa[(r + 1) >> 2], wb[(r + 1) >> 2], SEL[(r + 1) & 3]));
        E[r] = __viaddmax_s16x2(E[r], nEP, Ho[r]);                // E(i, j) = max(E(i, j-1) - e, H(i, j-1) - o)
        f = __viaddmax_s16x2(f, nEP, hup);                        // F(i, j) = max(F(i-1, j) - e, H(i-1, j) - o)
        Ho[r] = __vsub2(__vimax3_s16x2_relu(d, E[r], f), OP);     // H = max(0, diagonal, E, F)
        hup = Ho[r];
        if (r & 1) {
            rm[r >> 1] = __vimax3_s16x2(rm[r >> 1], Ho[r - 1], Ho[r]);
            cm = __vimax3_s16x2(cm, Ho[r - 1], Ho[r]);
        }
        d = dn;
    }
    return cm;
}

// A column that may hold a new end for one half (HI: the high one): the lane's largest Ho
// of the column and its first row, merged into the lane's best (larger Ho, then smaller
// row; a later column of the same row never replaces an earlier one), then the group's:
// its best and the first lane holding it.  Returns the value a cell of this lane must
// exceed to matter: the group's best for the lanes behind the holder, whose rows are
// larger, one less for the holder and the lanes before it, and never less than `none`, what
// a cell of H = 0 holds.  (A half without a pair has no other cells: one less than those,
// every later column called for this function, and the last grab of a run of 17 or 18 pairs took
// a third longer: 990 GCUPS at 60 residues and 18 pairs a query, 1,395 so; 1,623 and 2,138 at
// 120.)
template <int G, int LR, bool HI>
__device__ __forceinline__ int note_best(const uint32_t (&Ho)[LR], bool mine, int row0, int j, int lg, uint32_t sh16,
                                         int none, int &bv, int &brow, int &bcol) {
    int kk = (int)0x80000000;
#pragma unroll
    for (int r = 0; r < LR; ++r) {
        const uint32_t k = HI ? (Ho[r] & 0xFFFF0000u) | (uint32_t)(LR - 1 - r) : madd(Ho[r], sh16, (uint32_t)(LR - 1 - r));
        kk = max(kk, (int)k);
    }
    const int v = kk >> 16, row = row0 + LR - 1 - (kk & 0xFFFF);
    if (mine && (v > bv || (v == bv && row < brow))) { bv = v; brow = row; bcol = j; }
    int gk = bv * 64 + (63 - lg);
    for (int d = G >> 1; d > 0; d >>= 1) gk = max(gk, __shfl_xor_sync(0xffffffffu, gk, d));
    const int holder = 63 - (gk & 63);
    return max((gk >> 6) - (lg > holder ? 0 : 1), none);
}

// One group's two pairs in pass 1: targets, columns and the outputs.
struct pair_io {
    const uint8_t *tA, *tB;
    int nA, nB;
    int16_t *bmA, *bmB;                        // null: the half holds no pair of its own
};

// Pass 1 over the whole matrices of the warp's 32 / G groups, two pairs with the same
// query each: pair A (target tA, nA columns) in the low halves, pair B in the high halves.
// Lane l of a group owns LR consecutive query rows and at step s does column j = s - l,
// taking the row above from lane l-1; with several stripes (G = 32 only) a stripe's last row
// is handed on through buf.  Columns outside a target (before its first: the wavefront's
// ramp; past its last) use the pad residue, which scores -64 against every row: before
// the first column that leaves every state at its initial value, and past the last no cell
// reaches the best of a smaller row, so no step tests its range.  Every lane holds one
// column of the group's target window and takes the next window's when the step that
// needs it comes, so one shuffle per step gives each lane its column's residues.
// The end (the largest H, then the smallest row, then the smallest column) is kept per
// lane and looked at only in the steps whose column holds a value that can replace it
// (note_best): on random pairs 20 of 325 steps a pair; tracking each row's first maximum
// in a 32-bit key instead cost three integer-pipe and one multiply-add instruction per row.
// What bounds it is the integer pipe: per register and row prmt, two maxima for E and F, one
// for H and one for both running maxima, at half rate.  Measured (2.00e11 cells, 10^6
// pairs of 20,000 proteins with 25 substitutes): 69.6 ms with 32 lanes a pair, at most 16
// rows a lane and a key per row, 44.2 ms so (4,520 GCUPS); queries of 1,000 residues 43.7
// -> 25.3 ms.  A function of its own, so that what the caller keeps is saved around it
// instead of spilled inside its loop (1% faster).
// Writes bm[g] = the largest H on rows 2g and 2g+1 (pass 2's bound).
template <int G, int LR, bool MULTI>
__device__ __noinline__ void score_group(const uint8_t *__restrict__ prof, const sw_tile tl, const pair_io &io, int m, int o, int e,
                            uint32_t one, uint2 *buf, int sstride, end_cell *ra, end_cell *rb) {
    const int lg = threadIdx.x & (G - 1);
    const int n = __reduce_max_sync(0xffffffffu, max(io.nA, io.nB));
    constexpr int PLANE = G * SLOT, SBYTES = LR > SLOT ? 2 * PLANE : PLANE;
    const int nstripes = MULTI ? tl.ns : 1;
    const uint32_t INIT = ((uint32_t)(-o) & 0xFFFFu) * P2;  // -o in both halves
    const uint32_t OP = (uint32_t)o * P2, nEP = ((uint32_t)(-e) & 0xFFFFu) * P2;
    const uint32_t sh16 = one << 16;                        // 2^16 at run time (keeps the multiply-add)
    constexpr uint32_t PADS = (uint32_t)PAD_RES * P2;
    int vA = -o, iA = 0, jA = 0, vB = -o, iB = 0, jB = 0;   // the lane's best Ho, its row and column
    uint32_t tm = INIT;                                     // what a column must exceed to matter, per half
    for (int stripe = 0; stripe < nstripes; ++stripe) {
        const int row0 = (stripe * G + lg) * LR;
        uint32_t Ho[LR], E[LR], rm[LR / 2];
#pragma unroll
        for (int r = 0; r < LR; ++r) { Ho[r] = INIT; E[r] = INIT; rm[r >> 1] = INIT; }
        uint32_t hd = INIT;                                 // Ho(row0 - 1, j - 1)
        uint32_t out_h = INIT, out_f = INIT;
        const bool take = MULTI && stripe > 0, hand_on = MULTI && stripe + 1 < nstripes;
        const uint2 *in_buf = buf + (size_t)(stripe & 1) * sstride;
        uint2 *out_buf = buf + (size_t)((stripe + 1) & 1) * sstride;
        const uint8_t *pr = prof + stripe * SBYTES + lg * SLOT;
        if (take) {                                         // later rows must beat the earlier stripes' best
            int a = vA, b = vB;
            for (int d = G >> 1; d > 0; d >>= 1) {
                a = max(a, __shfl_xor_sync(0xffffffffu, a, d));
                b = max(b, __shfl_xor_sync(0xffffffffu, b, d));
            }
            tm = ((uint32_t)a & 0xFFFFu) | ((uint32_t)b << 16);
        }
        auto residues = [&](int x) {
            return (x < io.nA ? (uint32_t)io.tA[x] : (uint32_t)PAD_RES) |
                   ((x < io.nB ? (uint32_t)io.tB[x] : (uint32_t)PAD_RES) << 16);
        };
        uint32_t win = PADS, nxt = residues(lg);
        int j = -lg;
        const int steps = n + G - 1;
        for (int w = 0; w < steps; w += G) {
            const uint32_t cur = nxt;                       // columns [w, w + G)
            nxt = residues(w + G + lg);
            const int we = min(G, steps - w);
#pragma unroll 1
            for (int x = 0; x < we; ++x, ++j) {
                win = lg == x ? cur : win;
                const uint32_t tt = __shfl_sync(0xffffffffu, win, j, G);
                uint32_t hu = __shfl_up_sync(0xffffffffu, out_h, 1, G);
                uint32_t fu = __shfl_up_sync(0xffffffffu, out_f, 1, G);
                if (lg == 0) { hu = INIT; fu = INIT; }
                if (take && lg == 0 && j < n) { const uint2 v = in_buf[j]; hu = v.x; fu = v.y; }
                uint32_t f = fu, hup = hu;
                const uint32_t cm = column2<LR, PLANE>(pr + (int)(tt & 0xFFFFu) * tl.prow,
                                                       pr + (int)(tt >> 16) * tl.prow, Ho, E, rm, hd, f, hup, tm, OP, nEP);
                hd = hu;
                out_h = hup; out_f = f;
                if (hand_on && lg == G - 1 && (unsigned)j < (unsigned)n) out_buf[j] = make_uint2(hup, f);
                const uint32_t over = cm ^ tm;
                if (__builtin_expect(__any_sync(0xffffffffu, over != 0u), 0)) {
                    if (__any_sync(0xffffffffu, (over & 0xFFFFu) != 0u)) {
                        const int t = note_best<G, LR, false>(Ho, (over & 0xFFFFu) != 0u, row0, j, lg, sh16, -o, vA, iA,
                                                              jA);
                        tm = (tm & 0xFFFF0000u) | ((uint32_t)t & 0xFFFFu);
                    }
                    if (__any_sync(0xffffffffu, (over >> 16) != 0u)) {
                        const int t = note_best<G, LR, true>(Ho, (over >> 16) != 0u, row0, j, lg, sh16, -o, vB, iB, jB);
                        tm = (tm & 0xFFFFu) | ((uint32_t)t << 16);
                    }
                }
            }
        }
        // the row-pair bounds (LR is even, so no pair of rows straddles two lanes)
#pragma unroll
        for (int r = 0; r < LR; r += 2) {
            const int g = (row0 + r) >> 1;
            if (row0 + r < m) {
                const uint32_t h = __vadd2(rm[r >> 1], OP);
                if (io.bmA) io.bmA[g] = (int16_t)(h & 0xFFFFu);
                if (io.bmB) io.bmB[g] = (int16_t)(h >> 16);
            }
        }
        __syncwarp();
    }
    // across the group: the largest score, then the smallest row (rows are unique per lane)
    auto finish = [&](int v, int i, int j, end_cell *r) {
        int S = v;
        for (int d = G >> 1; d > 0; d >>= 1) S = max(S, __shfl_xor_sync(0xffffffffu, S, d));
        int bi = v == S ? i : 0x7FFFFFFF;
        for (int d = G >> 1; d > 0; d >>= 1) bi = min(bi, __shfl_xor_sync(0xffffffffu, bi, d));
        int bj = v == S && i == bi ? j : -1;
        for (int d = G >> 1; d > 0; d >>= 1) bj = max(bj, __shfl_xor_sync(0xffffffffu, bj, d));
        r->h = S + o; r->i = bi; r->j = bj;
    };
    finish(vA, iA, jA, ra);
    finish(vB, iB, jB, rb);
}

template <int G, bool MULTI>
__device__ __forceinline__ void score_rows(const sw_tile &tl, const uint8_t *prof, const pair_io &io, int m, int o,
                                           int e, uint32_t one, uint2 *buf, int sstride, end_cell *ea, end_cell *eb) {
#define PASTIS_SW_CASE(L) \
    case L: score_group<G, L, MULTI>(prof, tl, io, m, o, e, one, buf, sstride, ea, eb); break;
    switch (tl.lr) {
        PASTIS_SW_CASE(2) PASTIS_SW_CASE(4) PASTIS_SW_CASE(6) PASTIS_SW_CASE(8) PASTIS_SW_CASE(10)
        PASTIS_SW_CASE(12) PASTIS_SW_CASE(14) PASTIS_SW_CASE(16) PASTIS_SW_CASE(18) PASTIS_SW_CASE(20)
        PASTIS_SW_CASE(22) PASTIS_SW_CASE(24) PASTIS_SW_CASE(26) PASTIS_SW_CASE(28) PASTIS_SW_CASE(30)
        default: score_group<G, LR_MAX, MULTI>(prof, tl, io, m, o, e, one, buf, sstride, ea, eb); break;
    }
#undef PASTIS_SW_CASE
}

// ---------------------------------------------------------------------------------
// pass 2: bounding rectangle of the traced path, by an anchored DP over the reversed
// prefixes in which cells below a bound die
// ---------------------------------------------------------------------------------
// The suffix of the traced path that starts on forward row i scores S minus the
// forward value of the path state before it, which sits on row i-1; that value is at
// most bm[(i-1)/2], the largest H pass 1 saw on that pair of rows.  When the split
// falls inside a gap run, the reverse DP charges the suffix's part of the run an open
// instead of an extension, so its reverse value can be lower by o - e.  A reverse cell
// whose first row is i therefore dies below S - bm[(i-1)/2] - (o - e) (bm = 0 above
// row 0); every suffix of the path meets the bound, so the path survives, and the
// cells reaching S bound its begin.
// The band of an antidiagonal (a = rows back from the end, b = d - a columns back) is
// held two cells per lane, index k in lane k % 32 of chunk k / 32; the neighbours on
// the two antidiagonals before come by shuffles.  A live band wider than BAND cells
// returns false and the caller keeps the whole up-left rectangle.
constexpr int BAND = 64;
// Paths of at most this many rows take k_sw_carry (four rectangles a warp), longer ones with
// a row-by-row band k_sw_band.
constexpr int BAND_MIN_ROWS = 24;

// The value the previous antidiagonal holds at band index idx (NEG outside the band).
// `wide` is the same on every lane.
__device__ __forceinline__ int band_get(const int (&X)[2], int idx, bool wide) {
    const int v0 = __shfl_sync(0xffffffffu, X[0], idx & 31);
    int v = v0;
    if (wide) {
        const int v1 = __shfl_sync(0xffffffffu, X[1], idx & 31);
        v = idx >= 32 ? v1 : v0;
    }
    return (unsigned)idx < (wide ? 64u : 32u) ? v : NEG;
}

__device__ __noinline__ bool band_walk(const uint8_t *__restrict__ q, const uint8_t *__restrict__ t, const int *s_mat, int o,
                          int e, int S, int ei, int ej, const int16_t *__restrict__ bm, int *amax_out,
                          int *bmax_out) {
    const int lane = threadIdx.x & 31;
    const int A = ei + 1, B = ej + 1;
    const int slack = max(o - e, 0);
    int H1[2] = {lane == 0 ? 0 : NEG, NEG}, E1[2] = {NEG, NEG}, F1[2] = {NEG, NEG};   // d-1 (d = 0: the end)
    int H2[2] = {NEG, NEG};                                                          // d-2
    int w1 = 0, W1 = 1, w2 = 0, W2 = 0;            // band start and computed width of d-1, d-2
    int l1lo = 0, l1hi = 0, l2lo = 1, l2hi = 0;    // live ranges of a on d-1, d-2
    int amax = 0, bmax = 0;
    for (int d = 1; d <= A + B; ++d) {
        int clo = 0x7FFFFFFF, chi = -1;
        if (l1lo <= l1hi) { clo = l1lo; chi = l1hi + 1; }
        if (l2lo <= l2hi) { clo = min(clo, l2lo + 1); chi = max(chi, l2hi + 1); }
        if (chi < 0) break;                        // nothing live on d-1 or d-2
        clo = max(max(clo, d - B), 0);
        chi = min(min(chi, A), d);
        const int W = max(chi - clo + 1, 0);
        if (W > BAND) return false;
        const bool wide = W > 32 || W1 > 32 || W2 > 32;
        int h[2] = {NEG, NEG}, ev[2] = {NEG, NEG}, fv[2] = {NEG, NEG};
        unsigned live[2] = {0u, 0u};
        int ta = 0, tb = 0;                        // this lane's largest (a, b) reaching S
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            if (c == 1 && !wide) break;
            const int a = clo + 32 * c + lane, b = d - a;
            const int sa = a - w1, su = a - 1 - w1, s2 = a - 1 - w2;
            const int h1a = band_get(H1, sa, wide), e1a = band_get(E1, sa, wide);
            const int h1u = band_get(H1, su, wide), f1u = band_get(F1, su, wide);
            const int h2 = band_get(H2, s2, wide);
            if (a <= chi) {
                if (b >= 1) ev[c] = max(max(h1a - o, e1a - e), NEG);
                if (a >= 1) fv[c] = max(max(h1u - o, f1u - e), NEG);
                int dv = NEG;
                if (a >= 1 && b >= 1 && h2 != NEG)
                    dv = h2 + s_mat[(int)q[ei - (a - 1)] * PASTIS_NSYM + (int)t[ej - (b - 1)]];
                int hh = max(max(dv, ev[c]), fv[c]);
                const int i = ei - a + 1;          // first forward row of the suffix
                const int thr = S - (i >= 1 ? (int)bm[(i - 1) >> 1] : 0) - slack;
                if (hh < thr) { hh = NEG; ev[c] = NEG; fv[c] = NEG; }
                h[c] = hh;
                if (hh == S) { ta = a; tb = max(tb, b); }
            }
            live[c] = __ballot_sync(0xffffffffu, h[c] != NEG);
        }
        if (__any_sync(0xffffffffu, ta > 0 || tb > 0)) {
            amax = max(amax, __reduce_max_sync(0xffffffffu, ta));
            bmax = max(bmax, __reduce_max_sync(0xffffffffu, tb));
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) { H2[c] = H1[c]; H1[c] = h[c]; E1[c] = ev[c]; F1[c] = fv[c]; }
        w2 = w1; W2 = W1; w1 = clo; W1 = W;
        l2lo = l1lo; l2hi = l1hi;
        if (live[0] | live[1]) {
            l1lo = clo + (live[0] ? __ffs(live[0]) - 1 : 32 + __ffs(live[1]) - 1);
            l1hi = clo + (live[1] ? 63 - __clz(live[1]) : 31 - __clz(live[0]));
        } else {
            l1lo = 1; l1hi = 0;
        }
    }
    *amax_out = amax;
    *bmax_out = bmax;
    return true;
}

// The same reverse DP row by row, for o >= e.  The row's columns c0 .. lie in chunks of 32,
// lane L holding column c0 + 32 c + L of each: H, F and the target residue, which stay in
// their lanes from row to row, so that only the diagonal comes by shuffle; when moving the
// window to the first live column saves a chunk, the values are shifted there.  E along the
// row is an exclusive prefix maximum over the columns to the left, taken over max(D, F):
// with o >= e a gap that E itself opened never beats extending E, and as the threshold is
// the same along a row, a gap run through a cell below it stays below it; it is formed
// only when some cell is high enough for a gap opened there to stay alive.  So the live
// cells and their values are those of the antidiagonal form.  Returns false when a row
// needs more than ROW_COLS columns: near the begin of a path another alignment often holds
// the largest H of a row, the threshold is low, and some 60 to 100 columns stay alive.
// band[k] (null: not wanted) receives, for the forward rows ei - 8 k - 7 .. ei - 8 k, the
// first and the last (<< 16) column that the traced path can visit there: a diagonal step
// at forward cell (i, j) starts a suffix at reverse cell (a, b) = (ei - i + 1, ej - j + 1); a
// step of a vertical gap at (i, j) one at (a, b - 1), so the row's range reaches one column
// further left; a step of a horizontal gap one at (a - 1, b), so it takes in the range of
// the row below.
// Measured: 10^5 pairs of 1,000 residues 7.3 ms with the window moved every row, 64 columns
// and E formed always, 5.7 ms so; 10^6 pairs of 20,000 proteins 8.7 -> 7.5 ms.
constexpr int ROW_CHUNKS = 4;
constexpr int ROW_COLS = 32 * ROW_CHUNKS;

__device__ bool band_rows(const uint8_t *__restrict__ q, const uint8_t *__restrict__ t, const int *s_mat, int o,
                          int e, int S, int ei, int ej, const int16_t *__restrict__ bm, int *amax_out,
                          int *bmax_out, uint32_t *__restrict__ band) {
    const int lane = threadIdx.x & 31;
    const int A = ei + 1, B = ej + 1;
    const int slack = max(o - e, 0);
    int H[ROW_CHUNKS], F[ROW_CHUNKS], tc[ROW_CHUNKS];   // row a - 1, then row a; residue of column b
    int c0 = 0, plo = 0, phi = 0;                       // window start; live columns of row a - 1
    auto residue = [&](int b) { return b >= 1 && b <= B ? (int)t[ej - b + 1] : 0; };
    // row 0: the end (column 0), and the gaps opened from it
    const int thr0 = S - (int)bm[ei >> 1] - slack;
#pragma unroll
    for (int c = 0; c < ROW_CHUNKS; ++c) {
        const int b = 32 * c + lane;
        const int h = b == 0 ? 0 : (b <= B ? -o - (b - 1) * e : NEG);
        H[c] = h >= thr0 ? h : NEG;
        F[c] = NEG;
        tc[c] = residue(b);
        const unsigned live = __ballot_sync(0xffffffffu, H[c] != NEG);
        if (live) phi = 32 * c + 31 - __clz(live);
    }
    if (0 < thr0) plo = 1, phi = 0;                     // the end itself below its threshold
    else if (phi == ROW_COLS - 1 && -o - (ROW_COLS - 1) * e >= thr0 && ROW_COLS <= B) return false;
    int amax = 0, bmax = 0;
    int alive = 0;                                      // the last row with a live cell
    int blo = plo, bhi = phi;                           // live columns of the block's rows and the row below it
    auto put_band = [&](int k) {
        if (lane == 0) band[k] = (uint32_t)max(ej - bhi, 0) | (uint32_t)min(ej - blo + 1, ej) << 16;
    };
    for (int a = 1; a <= A && plo <= phi; ++a) {
        if (phi + 1 - plo >= ROW_COLS) return false;    // the diagonal successors leave the window
        if (((phi + 1 - plo) >> 5) < ((phi + 1 - c0) >> 5)) {
            const int sh = plo - c0, lane_to = (lane + sh) & 31;
            for (int x = sh >> 5; x > 0; --x) {         // whole chunks
#pragma unroll
                for (int c = 0; c < ROW_CHUNKS; ++c) {
                    H[c] = c + 1 < ROW_CHUNKS ? H[(c + 1) % ROW_CHUNKS] : NEG;
                    F[c] = c + 1 < ROW_CHUNKS ? F[(c + 1) % ROW_CHUNKS] : NEG;
                }
            }
            const bool own = lane + (sh & 31) < 32;
#pragma unroll
            for (int c = 0; c < ROW_CHUNKS; ++c) {
                const int h0 = __shfl_sync(0xffffffffu, H[c], lane_to), f0 = __shfl_sync(0xffffffffu, F[c], lane_to);
                int h1 = NEG, f1 = NEG;
                if (c + 1 < ROW_CHUNKS) {
                    h1 = __shfl_sync(0xffffffffu, H[(c + 1) % ROW_CHUNKS], lane_to);
                    f1 = __shfl_sync(0xffffffffu, F[(c + 1) % ROW_CHUNKS], lane_to);
                }
                H[c] = own ? h0 : h1;
                F[c] = own ? f0 : f1;
            }
            c0 = plo;
#pragma unroll
            for (int c = 0; c < ROW_CHUNKS; ++c) tc[c] = residue(c0 + 32 * c + lane);
        }
        const int i = ei - a + 1;                       // forward row of this reverse row
        const int thr = S - (i >= 1 ? (int)bm[(i - 1) >> 1] : 0) - slack;
        const int *row = s_mat + (int)q[i] * PASTIS_NSYM;
        int carry = NEG;                                // max of max(D, F) + k e left of the chunk
        int left = NEG;                                 // H of row a - 1 in the column before the chunk
        int tb = -1;                                    // this lane's largest column reaching S
        int nlo = 0x7FFFFFFF, nhi = -1;                 // live columns of this row
        bool more = false;
#pragma unroll
        for (int c = 0; c < ROW_CHUNKS; ++c) {
            // as far as row a - 1 reaches, or a gap run that stays at or above the threshold
            more = carry - o - (32 * c - 1) * e >= thr;
            if (phi + 1 < c0 + 32 * c && !more) break;
            const int k = 32 * c + lane, b = c0 + k;
            int hd = __shfl_up_sync(0xffffffffu, H[c], 1);
            if (lane == 0) hd = left;
            left = __shfl_sync(0xffffffffu, H[c], 31);
            int fv = max(max(H[c] - o, F[c] - e), NEG);
            int h = max(hd != NEG ? hd + row[tc[c]] : NEG, fv);
            if (b > B) h = NEG;
            if (more || __any_sync(0xffffffffu, h - o >= thr)) {
                int incl = h > NEG ? h + k * e : NEG;
#pragma unroll
                for (int x = 1; x < 32; x <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, x);
                    if (lane >= x) incl = max(incl, y);
                }
                int excl = __shfl_up_sync(0xffffffffu, incl, 1);
                if (lane == 0) excl = NEG;
                excl = max(excl, carry);
                carry = max(carry, __shfl_sync(0xffffffffu, incl, 31));
                if (excl > NEG && b <= B) h = max(h, excl - o - (k - 1) * e);
            }
            const bool dead = h < thr || b > B;
            H[c] = dead ? NEG : h;
            F[c] = dead ? NEG : fv;
            const unsigned live = __ballot_sync(0xffffffffu, !dead);
            if (live) {
                nlo = min(nlo, c0 + 32 * c + __ffs(live) - 1);
                nhi = c0 + 32 * c + 31 - __clz(live);
            }
            if (!dead && h == S) tb = b;
            if (c + 1 == ROW_CHUNKS) more = carry - o - (ROW_COLS - 1) * e >= thr;
            else more = false;
        }
        if (more) return false;                         // a run still going past the last chunk
        if (__any_sync(0xffffffffu, tb >= 0)) {
            amax = a;
            bmax = max(bmax, __reduce_max_sync(0xffffffffu, tb < 0 ? 0 : tb));
        }
        if (nhi >= 0) {
            plo = nlo; phi = nhi;
            blo = min(blo, plo);
            bhi = max(bhi, phi);
            alive = a;
            if ((a & 7) == 0) {
                if (band) put_band((a - 1) >> 3);
                blo = plo;
                bhi = phi;
            }
        } else {
            plo = 1; phi = 0;
        }
    }
    if (band && (alive & 7) != 0) put_band((alive - 1) >> 3);     // the last block, partly filled
    *amax_out = amax;
    *bmax_out = bmax;
    return true;
}

// Where the block ranges of pair p start (entries of bm_off are row pairs, four to a block;
// one more per pair covers the rounding).
__device__ __forceinline__ int64_t band_at(int64_t bm_off, int64_t p) { return (bm_off >> 2) + p; }

// Four lists of pairs in two arrays of one entry per pair: rings of 4 and 16 lanes from the
// two ends of the first, of 8 and 32 of the second.
constexpr int BAND_RINGS = 4;
__host__ __device__ __forceinline__ int64_t band_slot(int ring, int x, int64_t cap) {
    return (ring & 1) * cap + (ring < 2 ? x : cap - 1 - x);
}

// Whether a ring of G lanes can take the K blocks of a band in turn (k_sw_band): a lane
// that takes block b (in forward order) at steps column + b has to be done with it one step
// before the step at which block b + G, which it takes next, starts.
__device__ __forceinline__ bool band_fits(const uint32_t *band, int K, int G) {
    const int lane = threadIdx.x & 31;
    bool ok = true;
    for (int k = G + lane; k < K; k += 32)              // block k comes G blocks before block k - G
        ok &= (int)(band[k] >> 16) - (int)(band[k - G] & 0xFFFFu) < G - 1;
    return __all_sync(0xffffffffu, ok);
}

// Pass 2 over every pair pass 1 scored: one warp per pair, a few pairs per grab.
__global__ void __launch_bounds__(SW_THREADS, 5) k_sw_bound(const uint8_t *qcodes, const int64_t *qoffsets,
                                                         const uint8_t *tcodes, const int64_t *toffsets,
                                                         const pastis_cand *pairs, int64_t n_pairs,
                                                         const int8_t *gmat, int o, int e, const int16_t *bm_all,
                                                         const int64_t *bm_off, unsigned long long *next_pair,
                                                         sw_score_out *res, int cov_cut, uint32_t *band_all,
                                                         uint32_t *list, int64_t list_cap, int *n_band,
                                                         const int64_t *dn, const int *chk) {
    if (dn) n_pairs = *dn;
    if (chk && (chk[0] | chk[1])) return;
    __shared__ int s_mat[PASTIS_NSYM * PASTIS_NSYM];
    for (int x = threadIdx.x; x < PASTIS_NSYM * PASTIS_NSYM; x += blockDim.x) s_mat[x] = gmat[x];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    // eight pairs a grab, fewer when there are not enough for four grabs a warp
    const int64_t warps = (int64_t)gridDim.x * SW_WARPS;
    const int grab = (int)min((int64_t)8, max((int64_t)1, n_pairs / (4 * warps)));
    for (;;) {
        unsigned long long g = 0;
        if (lane == 0) g = atomicAdd(next_pair, (unsigned long long)grab);
        g = __shfl_sync(0xffffffffu, g, 0);
        if (g >= (unsigned long long)n_pairs) break;
        // lane u < grab fetches pair g + u's pass-1 result, sequences and bounds, so the
        // grab's load chains run side by side instead of one after the other
        int ok_l = 0, sc_l = 0, ei_l = 0, ej_l = 0, lq_l = 0, lt_l = 0;
        int64_t qo_l = 0, to_l = 0, bo_l = 0;
        const int64_t pl = (int64_t)g + lane;
        if (lane < grab && pl < n_pairs) {
            const sw_score_out r = res[pl];
            if (!r.big && r.score > 0) {
                const pastis_cand c = pairs[pl];
                qo_l = qoffsets[c.i];
                to_l = toffsets[c.j];
                bo_l = bm_off[pl];
                sc_l = r.score; ei_l = r.end_i; ej_l = r.end_j;
                lq_l = (int)(qoffsets[c.i + 1] - qo_l);
                lt_l = (int)(toffsets[c.j + 1] - to_l);
                // the filter-only mode: a pair whose end already rules out coverage
                ok_l = !(cov_cut >= 0 && cannot_cover(r, lq_l, lt_l, cov_cut));
            }
        }
        for (int u = 0; u < grab; ++u) {
            if (!__shfl_sync(0xffffffffu, ok_l, u)) continue;
            const int64_t p = (int64_t)g + u;
            const int score = __shfl_sync(0xffffffffu, sc_l, u);
            const int ei = __shfl_sync(0xffffffffu, ei_l, u), ej = __shfl_sync(0xffffffffu, ej_l, u);
            const uint8_t *qp = qcodes + __shfl_sync(0xffffffffu, qo_l, u);
            const uint8_t *tp = tcodes + __shfl_sync(0xffffffffu, to_l, u);
            const int64_t bo = __shfl_sync(0xffffffffu, bo_l, u);
            const int lq = __shfl_sync(0xffffffffu, lq_l, u), lt = __shfl_sync(0xffffffffu, lt_l, u);
            const int16_t *bm = bm_all + bo;
            uint32_t *band = band_all ? band_all + band_at(bo, p) : nullptr;
            int amax = 0, bmax = 0;
            bool ok = o >= e && band_rows(qp, tp, s_mat, o, e, score, ei, ej, bm, &amax, &bmax, band);
            const bool banded = ok && band;
            if (!ok) ok = band_walk(qp, tp, s_mat, o, e, score, ei, ej, bm, &amax, &bmax);
            if (ok && amax > 0 && bmax > 0) {      // else: the whole up-left rectangle (0, 0)
                sw_score_out r;
                r.end_i = ei; r.end_j = ej; r.rect_i = ei + 1 - amax; r.rect_j = ej + 1 - bmax;
                int ring = BAND_RINGS;             // the pair on a ring of 4 << ring lanes, if any
                if (banded && amax > BAND_MIN_ROWS && !(cov_cut >= 0 && cannot_cover(r, lq, lt, cov_cut))) {
                    __syncwarp();                  // lane 0 wrote the ranges
                    const int K = (amax + 7) >> 3;
                    ring = 0;
                    while (ring < BAND_RINGS && !band_fits(band, K, 4 << ring)) ++ring;
                }
                if (lane == 0) {
                    res[p].rect_i = r.rect_i;
                    res[p].rect_j = r.rect_j;
                    if (ring < BAND_RINGS) {
                        res[p].big = 2;
                        list[band_slot(ring, atomicAdd(&n_band[ring], 1), list_cap)] = (uint32_t)p;
                    }
                }
            }
        }
    }
}

// Row-pair bound entries of each pair: (query length + 1) / 2.
__global__ void k_bm_count(const pastis_cand *pairs, int64_t n, const int64_t *qoffsets, int64_t *cnt,
                           const int64_t *dn, const int *chk) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    // past the batch, or a batch the checks refused (its indexes are not to be followed)
    if ((dn && p >= *dn) || (chk && (chk[0] | chk[1]))) { cnt[p] = 0; return; }
    const int i = pairs[p].i;
    cnt[p] = (qoffsets[i + 1] - qoffsets[i] + 1) / 2;
}

__global__ void __launch_bounds__(SW_THREADS, 2) k_sw_score(const uint8_t *qcodes, const int64_t *qoffsets,
                                                         const uint8_t *tcodes, const int64_t *toffsets,
                                                         const pastis_cand *pairs, const int64_t *seg_start,
                                                         const uint32_t *seg_order, int64_t n_seg,
                                                         const int8_t *gmat, int o, int e,
                                                         int max_s, int prow_cap, uint32_t one, char *scratch,
                                                         size_t warp_bytes, int sstride, int *next_seg,
                                                         int16_t *bm_all, const int64_t *bm_off, sw_score_out *out,
                                                         unsigned long long *cells, const uint8_t *extra,
                                                         unsigned long long *tune, const uint32_t *d_nseg,
                                                         const int *chk) {
    // captured launches: the segment count from device memory, nothing on bad input
    if (d_nseg) n_seg = *d_nseg;
    if (chk && (chk[0] | chk[1])) return;
    // dynamic shared memory: the profile [NRES][prow_cap] bytes (prow_cap a whole number of
    // 512-row stripes); before it is built, the segment's sort keys
    extern __shared__ __align__(16) uint8_t s_prof[];
    __shared__ int s_seg, s_next;
    __shared__ uint16_t s_ord[SEG_MAX];
    uint32_t *s_key = reinterpret_cast<uint32_t *>(s_prof);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gw = blockIdx.x * SW_WARPS + warp;
    uint2 *my = reinterpret_cast<uint2 *>(scratch + (size_t)gw * warp_bytes);
    const bool packable = o <= GAP_MAX;
    unsigned long long my_cells = 0;
    for (;;) {
        if (threadIdx.x == 0) { s_seg = atomicAdd(next_seg, 1); s_next = 0; }
        __syncthreads();
        if (s_seg >= n_seg) break;
        const int64_t sg = seg_order[s_seg];
        const long long t_seg = tune ? clock64() : 0;
        const int64_t p0 = seg_start[sg], p1 = seg_start[sg + 1];
        const int cnt = (int)(p1 - p0);
        const int qi = pairs[p0].i;
        const int64_t qo = qoffsets[qi];
        const int m = (int)(qoffsets[qi + 1] - qo);
        const int bin = sw_bin(m);
        const bool int32_bin = extra[bin] == PASTIS_SW_INT32;    // the bin's pairs in 32-bit lanes
        // the segment's pairs by target length, longest first, so that the pairs of a warp
        // match and the last pairs taken are the shortest
        int np2 = 2;
        while (np2 < cnt) np2 <<= 1;
        for (int x = threadIdx.x; x < np2; x += SW_THREADS) {
            uint32_t key = 0xFFFFFFFFu;
            if (x < cnt) {
                const int j = pairs[p0 + x].j;
                key = ((uint32_t)(65535 - (toffsets[j + 1] - toffsets[j])) << 9) | (uint32_t)x;
            }
            s_key[x] = key;
        }
        __syncthreads();
        for (int k = 2; k <= np2; k <<= 1) {
            for (int jj = k >> 1; jj > 0; jj >>= 1) {
                for (int t = threadIdx.x; t < np2 / 2; t += SW_THREADS) {
                    const int x = 2 * t - (t & (jj - 1)), y = x + jj;
                    const uint32_t u = s_key[x], v = s_key[y];
                    if ((u > v) == ((x & k) == 0)) { s_key[x] = v; s_key[y] = u; }
                }
                __syncthreads();
            }
        }
        const int nt = 65535 - (int)(s_key[0] >> 9);
        for (int x = threadIdx.x; x < cnt; x += SW_THREADS) s_ord[x] = (uint16_t)(s_key[x] & (SEG_MAX - 1));
        const sw_tile tl = pick_tile(m, int32_bin ? 0 : extra[bin], cnt, nt, prow_cap);
        __syncthreads();
        // query profile: row i = (st * G + l) * lr + r of the query at byte
        // st * sbytes + (r / 16) * 16 G + 16 l + r % 16 of residue c = M[q_i][c] + o; o - 64
        // for the pad residue, unused slots and rows past the query
        if (tl.prow <= prow_cap) {
            const int gl = __ffs(tl.G) - 1, planes = tl.lr > SLOT ? 2 : 1;
            for (int x = threadIdx.x; x < tl.prow; x += SW_THREADS) {
                const int lq = (x >> 4) & (tl.G - 1), pl = x >> (4 + gl);
                const int st = planes == 2 ? pl >> 1 : pl, r = (planes == 2 ? (pl & 1) * SLOT : 0) + (x & 15);
                const int i = (st * tl.G + lq) * tl.lr + r;
                const bool in = r < tl.lr && i < m;
                const int8_t *row = gmat + (in ? (int)qcodes[qo + i] * PASTIS_NSYM : 0);
#pragma unroll
                for (int c = 0; c < NRES; ++c)
                    s_prof[c * tl.prow + x] = (uint8_t)(int8_t)(in && c < PASTIS_NSYM ? (int)row[c < PASTIS_NSYM ? c : 0] + o : o - 64);
            }
        }
        __syncthreads();
        const int grp = lane / tl.G, lg = lane & (tl.G - 1);
        for (;;) {
            int pk = 0;
            if (lane == 0) pk = atomicAdd(&s_next, 64 / tl.G);
            pk = __shfl_sync(0xffffffffu, pk, 0);
            if (pk >= cnt) break;
            pk += 2 * grp;
            int64_t pp[2];
            int nn[2], st[2];                                     // st: 0 zero, 1 big, 2 run
            const uint8_t *tp[2];
            for (int u = 0; u < 2; ++u) {
                pp[u] = pk + u < cnt ? p0 + (int64_t)s_ord[pk + u] : -1;
                nn[u] = 0; st[u] = 0; tp[u] = tcodes;
                if (pp[u] < 0) continue;
                const pastis_cand c = pairs[pp[u]];
                const int64_t to = toffsets[c.j];
                nn[u] = (int)(toffsets[c.j + 1] - to);
                tp[u] = tcodes + to;
                if (m == 0 || nn[u] == 0) st[u] = 0;
                else if (int32_bin || !packable || tl.prow > prow_cap ||
                         (int64_t)max_s * (int64_t)min(m, nn[u]) >= SCORE_MAX) st[u] = 1;
                else st[u] = 2;
            }
            end_cell ea, eb;
            ea.h = eb.h = 0;
            ea.i = ea.j = eb.i = eb.j = 0;
            if (__any_sync(0xffffffffu, st[0] == 2 || st[1] == 2)) {
                pair_io io;
                io.tA = tp[0]; io.tB = tp[1];
                io.nA = st[0] == 2 ? nn[0] : 0;                   // a half without a pair runs on pad columns
                io.nB = st[1] == 2 ? nn[1] : 0;
                io.bmA = st[0] == 2 ? bm_all + bm_off[pp[0]] : nullptr;
                io.bmB = st[1] == 2 ? bm_all + bm_off[pp[1]] : nullptr;
                // one loop body per lane count and rows per lane, and for several stripes: with
                // the lane count and the hand-on as run-time values pass 1 took 6% longer
                if (tl.ns > 1) score_rows<32, true>(tl, s_prof, io, m, o, e, one, my, sstride, &ea, &eb);
                else if (tl.G == 32) score_rows<32, false>(tl, s_prof, io, m, o, e, one, my, sstride, &ea, &eb);
                else if (tl.G == 16) score_rows<16, false>(tl, s_prof, io, m, o, e, one, my, sstride, &ea, &eb);
                else score_rows<8, false>(tl, s_prof, io, m, o, e, one, my, sstride, &ea, &eb);
                __syncwarp();
            }
            if (lg == 0) {
                for (int u = 0; u < 2; ++u) {
                    if (pp[u] < 0) continue;
                    const end_cell &en = u ? eb : ea;
                    sw_score_out r;
                    r.score = 0; r.end_i = 0; r.end_j = 0; r.rect_i = 0; r.rect_j = 0; r.big = st[u] == 1;
                    if (st[u] == 2) {
                        if (en.h > 0) { r.score = en.h; r.end_i = en.i; r.end_j = en.j; }
                        my_cells += (unsigned long long)m * (unsigned long long)nn[u];
                    }
                    out[pp[u]] = r;
                }
            }
        }
        __syncthreads();
        if (tune && threadIdx.x == 0) atomicAdd(&tune[bin], (unsigned long long)(clock64() - t_seg));
    }
    if (cells && my_cells) atomicAdd(cells, my_cells);
}

// ---------------------------------------------------------------------------------
// pass 3: carries over the rectangle (or the whole matrix for very large scores)
// ---------------------------------------------------------------------------------
constexpr int CR = 8;                  // rows per lane of the small-rectangle groups and of TRACK

struct stripe3_cell { int32_t h, f; uint32_t hb, fb, hm, fm; };

__device__ __forceinline__ uint32_t pack_rc(int r, int c) { return ((uint32_t)r << 16) | (uint32_t)c; }

// Carries begin (row << 16 | col, of the first column) and identities << 16 | matched
// columns, with CR rows per lane (a stripe is 32 * CR rows).  TRACK: also finds the
// row-major first maximum (for pairs pass 1 skipped); otherwise reports the state at
// (m-1, n-1).
template <bool TRACK, int CR>
__device__ void carry_warp(const uint8_t *__restrict__ q, int m, const uint8_t *__restrict__ t, int n,
                           const int *__restrict__ s_mat, int o, int e, stripe3_cell *scratch, int sstride,
                           int *h_out, int *ei_out, int *ej_out, uint32_t *beg_out, uint32_t *im_out) {
    const int lane = threadIdx.x & 31;
    int best = 0, brow = 0x7FFFFFFF, bcol = 0;
    uint32_t bbeg = 0, bim = 0;
    int endh = NEG;
    uint32_t endb = 0, endm = 0;
    constexpr int STRIPE = 32 * CR;
    const int nstripes = (m + STRIPE - 1) / STRIPE;
    for (int stripe = 0; stripe < nstripes; ++stripe) {
        const int row0 = stripe * STRIPE + lane * CR;
        int qoff[CR], Hc[CR], Ec[CR];
        uint32_t HB[CR], EB[CR], HM[CR], EM[CR];
#pragma unroll
        for (int r = 0; r < CR; ++r) {
            const int i = row0 + r;
            qoff[r] = (i < m ? (int)q[i] : PASTIS_NSYM) * 32;
            Hc[r] = 0; Ec[r] = NEG;
            HB[r] = pack_rc(i + 1, 0); EB[r] = 0; HM[r] = 0; EM[r] = 0;
        }
        int dh = 0;
        uint32_t db = pack_rc(row0, 0), dm = 0;
        int out_h = 0, out_f = NEG, out_t = 0;
        uint32_t out_hb = 0, out_fb = 0, out_hm = 0, out_fm = 0;
        const stripe3_cell *in_buf = scratch + (size_t)(stripe & 1) * sstride;
        stripe3_cell *out_buf = scratch + (size_t)((stripe + 1) & 1) * sstride;
        const bool last = stripe + 1 == nstripes;
        for (int s = 0; s < n + 31; ++s) {
            const int j = s - lane;
            int up_h = __shfl_up_sync(0xffffffffu, out_h, 1);
            int up_f = __shfl_up_sync(0xffffffffu, out_f, 1);
            uint32_t up_hb = __shfl_up_sync(0xffffffffu, out_hb, 1);
            uint32_t up_fb = __shfl_up_sync(0xffffffffu, out_fb, 1);
            uint32_t up_hm = __shfl_up_sync(0xffffffffu, out_hm, 1);
            uint32_t up_fm = __shfl_up_sync(0xffffffffu, out_fm, 1);
            int tj = __shfl_up_sync(0xffffffffu, out_t, 1);
            if (lane == 0 && j < n) {
                tj = t[j];
                if (stripe == 0) {
                    up_h = 0; up_f = NEG; up_hb = pack_rc(0, j + 1); up_fb = 0; up_hm = 0; up_fm = 0;
                } else {
                    const stripe3_cell c = in_buf[j];
                    up_h = c.h; up_f = c.f; up_hb = c.hb; up_fb = c.fb; up_hm = c.hm; up_fm = c.fm;
                }
            }
            if (j >= 0 && j < n) {
                int ph = dh;
                uint32_t pb = db, pm = dm;
                int ah = up_h, f = up_f;
                uint32_t ab = up_hb, am = up_hm, fb = up_fb, fm = up_fm;
#pragma unroll
                for (int r = 0; r < CR; ++r) {
                    const int i = row0 + r;
                    const int eo = Hc[r] - o, ex = Ec[r] - e;
                    const bool eop = eo >= ex;
                    const int ev = eop ? eo : ex;
                    const uint32_t evb = eop ? HB[r] : EB[r], evm = eop ? HM[r] : EM[r];
                    const int fo = ah - o, fx = f - e;
                    const bool fop = fo >= fx;
                    f = fop ? fo : fx;
                    fb = fop ? ab : fb;
                    fm = fop ? am : fm;
                    int h = ph + s_mat[qoff[r] + tj];
                    uint32_t hb = pb, hm = pm + ((qoff[r] == tj * 32) ? 0x10001u : 1u);
                    if (f > h) { h = f; hb = fb; hm = fm; }
                    if (ev > h) { h = ev; hb = evb; hm = evm; }
                    if (h <= 0) { h = 0; hb = pack_rc(i + 1, j + 1); hm = 0; }
                    if (TRACK) {
                        if (i < m && (h > best || (h == best && h > 0 && i < brow))) {
                            best = h; brow = i; bcol = j; bbeg = hb; bim = hm;
                        }
                    } else if (i == m - 1 && j == n - 1) {
                        endh = h; endb = hb; endm = hm;
                    }
                    ph = Hc[r]; pb = HB[r]; pm = HM[r];
                    Hc[r] = h; HB[r] = hb; HM[r] = hm;
                    Ec[r] = ev; EB[r] = evb; EM[r] = evm;
                    ah = h; ab = hb; am = hm;
                }
                dh = up_h; db = up_hb; dm = up_hm;
                out_h = ah; out_f = f; out_t = tj;
                out_hb = ab; out_fb = fb; out_hm = am; out_fm = fm;
                if (lane == 31 && !last) out_buf[j] = stripe3_cell{ah, f, ab, fb, am, fm};
            }
        }
        __syncwarp();
    }
    if (TRACK) {
        for (int d = 16; d > 0; d >>= 1) {
            const int ob = __shfl_xor_sync(0xffffffffu, best, d);
            const int orow = __shfl_xor_sync(0xffffffffu, brow, d);
            const int ocol = __shfl_xor_sync(0xffffffffu, bcol, d);
            const uint32_t obb = __shfl_xor_sync(0xffffffffu, bbeg, d);
            const uint32_t obm = __shfl_xor_sync(0xffffffffu, bim, d);
            if (ob > best || (ob == best && (orow < brow || (orow == brow && ocol < bcol)))) {
                best = ob; brow = orow; bcol = ocol; bbeg = obb; bim = obm;
            }
        }
        *h_out = best; *ei_out = brow; *ej_out = bcol; *beg_out = bbeg; *im_out = bim;
    } else {
        for (int d = 16; d > 0; d >>= 1) {
            const int oh = __shfl_xor_sync(0xffffffffu, endh, d);
            const uint32_t ob = __shfl_xor_sync(0xffffffffu, endb, d);
            const uint32_t om = __shfl_xor_sync(0xffffffffu, endm, d);
            if (oh > endh) { endh = oh; endb = ob; endm = om; }
        }
        *h_out = endh; *beg_out = endb; *im_out = endm;
    }
}

// Small rectangles (at most 64 rows): four per warp, each on an 8-lane group with 8
// rows per lane, all groups stepping together (the longest sets the step count) and
// shuffling within their 8 lanes.  Reports the state at each rectangle's last cell.
constexpr int GL = 8;                  // lanes per group
constexpr int GROWS = GL * CR;         // rows per group

__device__ void carry_group(const uint8_t *__restrict__ q, int m, const uint8_t *__restrict__ t, int n,
                            const int *__restrict__ s_mat, int o, int e, int *h_out, uint32_t *beg_out,
                            uint32_t *im_out) {
    const int lane = threadIdx.x & 31, lg = lane & (GL - 1);
    const int row0 = lg * CR;
    int qoff[CR], Hc[CR], Ec[CR];
    uint32_t HB[CR], EB[CR], HM[CR], EM[CR];
#pragma unroll
    for (int r = 0; r < CR; ++r) {
        const int i = row0 + r;
        qoff[r] = (i < m ? (int)q[i] : PASTIS_NSYM) * 32;
        Hc[r] = 0; Ec[r] = NEG;
        HB[r] = pack_rc(i + 1, 0); EB[r] = 0; HM[r] = 0; EM[r] = 0;
    }
    int dh = 0;
    uint32_t db = pack_rc(row0, 0), dm = 0;
    int out_h = 0, out_f = NEG, out_t = 0;
    uint32_t out_hb = 0, out_fb = 0, out_hm = 0, out_fm = 0;
    int endh = NEG;
    uint32_t endb = 0, endm = 0;
    const int nsteps = __reduce_max_sync(0xffffffffu, n > 0 ? n + GL - 1 : 0);
    for (int s = 0; s < nsteps; ++s) {
        const int j = s - lg;
        int up_h = __shfl_up_sync(0xffffffffu, out_h, 1, GL);
        int up_f = __shfl_up_sync(0xffffffffu, out_f, 1, GL);
        uint32_t up_hb = __shfl_up_sync(0xffffffffu, out_hb, 1, GL);
        uint32_t up_fb = __shfl_up_sync(0xffffffffu, out_fb, 1, GL);
        uint32_t up_hm = __shfl_up_sync(0xffffffffu, out_hm, 1, GL);
        uint32_t up_fm = __shfl_up_sync(0xffffffffu, out_fm, 1, GL);
        int tj = __shfl_up_sync(0xffffffffu, out_t, 1, GL);
        if (lg == 0 && j < n) {
            tj = t[j];
            up_h = 0; up_f = NEG; up_hb = pack_rc(0, j + 1); up_fb = 0; up_hm = 0; up_fm = 0;
        }
        if (j >= 0 && j < n) {
            int ph = dh;
            uint32_t pb = db, pm = dm;
            int ah = up_h, f = up_f;
            uint32_t ab = up_hb, am = up_hm, fb = up_fb, fm = up_fm;
#pragma unroll
            for (int r = 0; r < CR; ++r) {
                const int i = row0 + r;
                const int eo = Hc[r] - o, ex = Ec[r] - e;
                const bool eop = eo >= ex;
                const int ev = eop ? eo : ex;
                const uint32_t evb = eop ? HB[r] : EB[r], evm = eop ? HM[r] : EM[r];
                const int fo = ah - o, fx = f - e;
                const bool fop = fo >= fx;
                f = fop ? fo : fx;
                fb = fop ? ab : fb;
                fm = fop ? am : fm;
                int h = ph + s_mat[qoff[r] + tj];
                uint32_t hb = pb, hm = pm + ((qoff[r] == tj * 32) ? 0x10001u : 1u);
                if (f > h) { h = f; hb = fb; hm = fm; }
                if (ev > h) { h = ev; hb = evb; hm = evm; }
                if (h <= 0) { h = 0; hb = pack_rc(i + 1, j + 1); hm = 0; }
                if (i == m - 1 && j == n - 1) { endh = h; endb = hb; endm = hm; }
                ph = Hc[r]; pb = HB[r]; pm = HM[r];
                Hc[r] = h; HB[r] = hb; HM[r] = hm;
                Ec[r] = ev; EB[r] = evb; EM[r] = evm;
                ah = h; ab = hb; am = hm;
            }
            dh = up_h; db = up_hb; dm = up_hm;
            out_h = ah; out_f = f; out_t = tj;
            out_hb = ab; out_fb = fb; out_hm = am; out_fm = fm;
        }
    }
    for (int d = GL / 2; d > 0; d >>= 1) {
        const int oh = __shfl_xor_sync(0xffffffffu, endh, d, GL);
        const uint32_t ob = __shfl_xor_sync(0xffffffffu, endb, d, GL);
        const uint32_t om = __shfl_xor_sync(0xffffffffu, endm, d, GL);
        if (oh > endh) { endh = oh; endb = ob; endm = om; }
    }
    *h_out = endh; *beg_out = endb; *im_out = endm;
}

__device__ void finish_record(pastis_aln &rec, int S, int ei, int ej, int qb, int tb, int ident, int M, int lq,
                              int lt, int ani, int cov, int filtered) {
    rec.score = S;
    rec.qb = (uint16_t)qb; rec.qe = (uint16_t)(ei + 1); rec.tb = (uint16_t)tb; rec.te = (uint16_t)(ej + 1);
    rec.ident = (uint16_t)ident;
    rec.cols = (uint16_t)((ei + 1 - qb) + (ej + 1 - tb) - M);
    const int span = lq <= lt ? ei + 1 - qb : ej + 1 - tb;
    const int L = lq <= lt ? lq : lt;
    rec.passes = (rec.cols > 0 && 100 * ident >= ani * (int)rec.cols && 100 * span >= cov * L) ? 1 : 0;
    if (filtered && !rec.passes) { rec.qb = rec.tb = 0; rec.ident = rec.cols = 0; }
}

// Pass 3 inside a band: the pairs whose path pass 2 bounded row by row, a pair on a ring of
// G lanes.  The rows from the end upwards lie in blocks of 8; a lane takes blocks l, l + G,
// ... of the K blocks in forward order, block b at column c in step c + b, only over the
// columns pass 2 left it.  The row above a block comes by shuffle from the lane before it in
// the ring, which did that column one step earlier.  Cells outside the band count as
// zero cells a path may start after (no forward value is below zero, so no value inside
// exceeds the true one), and the band holds the traced path, so along it the values and
// choices are the traceback's.  What bounds it is instruction issue, 30 a cell; a band of
// some 25 columns a row instead of the whole rectangle leaves a tenth of the cells of two
// homologous proteins.  Pass 3 of the benchmark recipe at 5,000 proteins (1.18 M pairs, 97,000
// traced) 35.6 ms over the rectangles, 4.2 ms so; of 10^5 pairs of 1,000 residues 33.3 ->
// 3.5 ms; of 1,000 proteins (15,000 pairs, where the slowest warp counts) 9.1 -> 0.93 ms.

struct band_args {
    const uint8_t *qcodes;
    const int64_t *qoffsets;
    const uint8_t *tcodes;
    const int64_t *toffsets;
    const pastis_cand *pairs;
    int o, e, ani, cov, filtered;
    const uint32_t *band_all;
    const int64_t *bm_off;
    const uint32_t *list;
    int64_t list_cap;
    const int *n_list;
    int *next;
    const sw_score_out *res;
    pastis_aln *out;
    int *err;
};

template <int G>
__device__ __noinline__ void band_ring(const band_args &g, const int *s_mat) {
    const int o = g.o, e = g.e;
    const int lane = threadIdx.x & 31, lg = lane & (G - 1), from = (lane & ~(G - 1)) | ((lane + G - 1) & (G - 1));
    constexpr int RING = G == 4 ? 0 : (G == 8 ? 1 : (G == 16 ? 2 : 3));
    const int cnt = g.n_list[RING];
    int *const next = g.next + RING;
    // the group's pair
    bool busy = false, done = false;
    int64_t p = 0;
    const uint8_t *q = g.qcodes, *t = g.tcodes;
    const uint32_t *band = g.band_all;
    int K = 0, top = 0, ei = 0, ej = 0, rj = 0, step = 0;
    // the lane's block: rows row0 .. row0 + 7, columns lo .. hi; plo .. phi those of the block above
    int b = 0, row0 = 0, lo = 1, hi = 0, plo = 1, phi = 0;
    int qoff[8], Hc[8], Ec[8];
    uint32_t HB[8], EB[8], HM[8], EM[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) { qoff[r] = 0; Hc[r] = 0; Ec[r] = NEG; HB[r] = EB[r] = HM[r] = EM[r] = 0u; }
    int dh = 0, out_h = 0, out_f = NEG;
    uint32_t db = 0u, dm = 0u, out_hb = 0u, out_fb = 0u, out_hm = 0u, out_fm = 0u;
    auto open_block = [&]() {
        if (b >= K) { lo = 1; hi = 0; return; }
        const uint32_t own = band[K - 1 - b], above = b > 0 ? band[K - b] : 1u;
        lo = max((int)(own & 0xFFFFu), rj); hi = (int)(own >> 16);
        plo = max((int)(above & 0xFFFFu), b > 0 ? rj : 1); phi = (int)(above >> 16);
        row0 = top + 8 * b;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            qoff[r] = (row0 + r >= 0 ? (int)q[row0 + r] : PASTIS_NSYM) * 32;
            Hc[r] = 0; Ec[r] = NEG;
            HB[r] = pack_rc(row0 + r + 1, lo); EB[r] = 0u; HM[r] = 0u; EM[r] = 0u;
        }
    };
    for (;;) {
        if (__any_sync(0xffffffffu, !busy && !done)) {
            int slot = 0;
            if (!busy && !done && lg == 0) slot = atomicAdd(next, 1);
            slot = __shfl_sync(0xffffffffu, slot, lane & ~(G - 1));
            int t0 = 0x7FFFFFFF;
            const bool take = !busy && !done && slot < cnt;
            if (!busy && !done && slot >= cnt) done = true;
            if (take) {
                p = g.list[band_slot(RING, slot, g.list_cap)];
                const pastis_cand c = g.pairs[p];
                const sw_score_out r = g.res[p];
                q = g.qcodes + g.qoffsets[c.i];
                t = g.tcodes + g.toffsets[c.j];
                band = g.band_all + band_at(g.bm_off[p], p);
                ei = r.end_i; ej = r.end_j; rj = r.rect_j;
                K = (ei + 1 - r.rect_i + 7) >> 3;
                top = ei + 1 - 8 * K;
                b = lg;
                open_block();
                busy = true;
                if (b < K) t0 = lo + b - 1;
            }
#pragma unroll
            for (int d = G >> 1; d > 0; d >>= 1) t0 = min(t0, __shfl_xor_sync(0xffffffffu, t0, d));
            if (take) step = t0;
            if (__all_sync(0xffffffffu, done)) break;
        }
        // the row above at this lane's column, from the lane before it in the ring
        int up_h = __shfl_sync(0xffffffffu, out_h, from), up_f = __shfl_sync(0xffffffffu, out_f, from);
        uint32_t up_hb = __shfl_sync(0xffffffffu, out_hb, from), up_fb = __shfl_sync(0xffffffffu, out_fb, from);
        uint32_t up_hm = __shfl_sync(0xffffffffu, out_hm, from), up_fm = __shfl_sync(0xffffffffu, out_fm, from);
        const int c = step - b;
        if (c < plo || c > phi) { up_h = 0; up_f = NEG; up_hb = pack_rc(row0, c + 1); up_fb = 0u; up_hm = 0u; up_fm = 0u; }
        if (busy && c >= lo && c <= hi) {
            const int tj = t[c];
            int ph = dh, ah = up_h, f = up_f;
            uint32_t pb = db, pm = dm, ab = up_hb, am = up_hm, fb = up_fb, fm = up_fm;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int eo = Hc[r] - o, ex = Ec[r] - e;
                const bool eop = eo >= ex;
                const int ev = eop ? eo : ex;
                const uint32_t evb = eop ? HB[r] : EB[r], evm = eop ? HM[r] : EM[r];
                const int fo = ah - o, fx = f - e;
                const bool fop = fo >= fx;
                f = fop ? fo : fx;
                fb = fop ? ab : fb;
                fm = fop ? am : fm;
                int h = ph + s_mat[qoff[r] + tj];
                uint32_t hb = pb, hm = pm + ((qoff[r] == tj * 32) ? 0x10001u : 1u);
                if (f > h) { h = f; hb = fb; hm = fm; }
                if (ev > h) { h = ev; hb = evb; hm = evm; }
                if (h <= 0) { h = 0; hb = pack_rc(row0 + r + 1, c + 1); hm = 0u; }
                ph = Hc[r]; pb = HB[r]; pm = HM[r];
                Hc[r] = h; HB[r] = hb; HM[r] = hm;
                Ec[r] = ev; EB[r] = evb; EM[r] = evm;
                ah = h; ab = hb; am = hm;
            }
            out_h = ah; out_f = f; out_hb = ab; out_fb = fb; out_hm = am; out_fm = fm;
            if (b == K - 1 && c == ej) {           // the end: the last row of the last block
                const sw_score_out r1 = g.res[p];
                const pastis_cand cd = g.pairs[p];
                const int lq = (int)(g.qoffsets[cd.i + 1] - g.qoffsets[cd.i]);
                const int lt = (int)(g.toffsets[cd.j + 1] - g.toffsets[cd.j]);
                if (Hc[7] != r1.score) atomicExch(g.err, 1);
                pastis_aln rec;
                rec.seed_used = 0; rec.passes = 0; rec.reserved = 0;
                finish_record(rec, r1.score, ei, ej, (int)(HB[7] >> 16), (int)(HB[7] & 0xFFFFu), (int)(HM[7] >> 16),
                              (int)(HM[7] & 0xFFFFu), lq, lt, g.ani, g.cov, g.filtered);
                g.out[p] = rec;
            }
            if (c == hi) { b += G; open_block(); }
        }
        dh = up_h; db = up_hb; dm = up_hm;
        if (busy && step == ej + K - 1) busy = false;   // the same step for the whole group
        ++step;
    }
}

// The widest bands, of which there are few, first; a warp that finds a list empty goes on
// to the next, so the lists' last pairs run beside the next list's.
__global__ void __launch_bounds__(SW_THREADS, 2) k_sw_band(band_args g, const int8_t *gmat, const int *chk) {
    if (chk && (chk[0] | chk[1])) return;
    __shared__ int s_mat[(PASTIS_NSYM + 1) * 32];
    for (int x = threadIdx.x; x < (PASTIS_NSYM + 1) * 32; x += blockDim.x) {
        const int a = x / 32, b = x % 32;
        s_mat[x] = (a < PASTIS_NSYM && b < PASTIS_NSYM) ? (int)gmat[a * PASTIS_NSYM + b] : PAD_SCORE;
    }
    __syncthreads();
    band_ring<32>(g, s_mat);
    band_ring<16>(g, s_mat);
    band_ring<8>(g, s_mat);
    band_ring<4>(g, s_mat);
}

__global__ void __launch_bounds__(SW_THREADS) k_sw_carry(const uint8_t *qcodes, const int64_t *qoffsets,
                                                         const uint8_t *tcodes, const int64_t *toffsets,
                                                         const pastis_cand *pairs, int64_t n_pairs,
                                                         const int8_t *gmat, int o, int e, int ani, int cov,
                                                         stripe3_cell *scratch, int sstride, int *next_pair,
                                                         const sw_score_out *res, int score_only, int filtered,
                                                         pastis_aln *out,
                                                         int *err, unsigned long long *cells,
                                                         unsigned long long *tune, const int64_t *dn,
                                                         const int *chk) {
    if (dn) n_pairs = *dn;
    if (chk && (chk[0] | chk[1])) return;
    __shared__ int s_mat[(PASTIS_NSYM + 1) * 32];
    for (int x = threadIdx.x; x < (PASTIS_NSYM + 1) * 32; x += blockDim.x) {
        const int a = x / 32, b = x % 32;
        s_mat[x] = (a < PASTIS_NSYM && b < PASTIS_NSYM) ? (int)gmat[a * PASTIS_NSYM + b] : PAD_SCORE;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, grp = lane / GL, lg = lane & (GL - 1);
    const int gw = blockIdx.x * SW_WARPS + (threadIdx.x >> 5);
    stripe3_cell *my = scratch + (size_t)gw * 2 * sstride;
    unsigned long long my_cells = 0;
    for (;;) {
        int p0 = 0;
        if (lane == 0) p0 = atomicAdd(next_pair, 32 / GL);
        p0 = __shfl_sync(0xffffffffu, p0, 0);
        if (p0 >= n_pairs) break;
        // the four pairs of this warp: small rectangles go to the groups together
        const int64_t pg = p0 + grp;
        int gm = 0, gn = 0;
        const uint8_t *gq = qcodes, *gt = tcodes;
        sw_score_out g1;
        g1.score = 0; g1.big = 0; g1.end_i = g1.end_j = g1.rect_i = g1.rect_j = 0;
        if (pg < n_pairs) {
            g1 = res[pg];
            if (!score_only && !g1.big && g1.score > 0 && g1.end_i + 1 - g1.rect_i <= GROWS) {
                const pastis_cand c = pairs[pg];
                const bool skip = filtered && cannot_cover(g1, (int)(qoffsets[c.i + 1] - qoffsets[c.i]),
                                                           (int)(toffsets[c.j + 1] - toffsets[c.j]), cov);
                if (!skip) {                       // a skipped pair's record comes from the loop below
                    gm = g1.end_i + 1 - g1.rect_i;
                    gn = g1.end_j + 1 - g1.rect_j;
                    gq = qcodes + qoffsets[c.i] + g1.rect_i;
                    gt = tcodes + toffsets[c.j] + g1.rect_j;
                }
            }
        }
        int gh;
        uint32_t gb, gim;
        carry_group(gq, gm, gt, gn, s_mat, o, e, &gh, &gb, &gim);
        if (lg == 0 && pg < n_pairs && gm > 0) {
            const pastis_cand c = pairs[pg];
            const int lq = (int)(qoffsets[c.i + 1] - qoffsets[c.i]), lt = (int)(toffsets[c.j + 1] - toffsets[c.j]);
            if (gh != g1.score) atomicExch(err, 1);
            pastis_aln rec;
            rec.seed_used = 0; rec.passes = 0; rec.reserved = 0;
            finish_record(rec, g1.score, g1.end_i, g1.end_j, g1.rect_i + (int)(gb >> 16), g1.rect_j + (int)(gb & 0xFFFF),
                          (int)(gim >> 16), (int)(gim & 0xFFFF), lq, lt, ani, cov, filtered);
            out[pg] = rec;
        }
        // the others, one warp each
        for (int k = 0; k < 32 / GL; ++k) {
            const int64_t p = p0 + k;
            if (p >= n_pairs) break;
            const sw_score_out r1 = res[p];
            if (r1.big == 2) continue;             // k_sw_band's
            const pastis_cand c = pairs[p];
            const int64_t qo = qoffsets[c.i], to = toffsets[c.j];
            const int lq = (int)(qoffsets[c.i + 1] - qo), lt = (int)(toffsets[c.j + 1] - to);
            const bool skip = filtered && !r1.big && r1.score > 0 && cannot_cover(r1, lq, lt, cov);
            const bool small = !score_only && !r1.big && r1.score > 0 && r1.end_i + 1 - r1.rect_i <= GROWS;
            if (small && !skip) continue;
            pastis_aln rec;
            rec.score = 0; rec.qb = rec.qe = rec.tb = rec.te = 0; rec.ident = rec.cols = 0;
            rec.seed_used = 0; rec.passes = 0; rec.reserved = 0;
            if (r1.big) {
                const long long t_big = tune ? clock64() : 0;      // the tuner's cycles of 32-bit work
                if (lq > 0 && lt > 0) {
                    int h, bi, bj;
                    uint32_t beg, im;
                    carry_warp<true, CR>(qcodes + qo, lq, tcodes + to, lt, s_mat, o, e, my, sstride, &h, &bi, &bj, &beg,
                                         &im);
                    if (h > 0)
                        finish_record(rec, h, bi, bj, (int)(beg >> 16), (int)(beg & 0xFFFF), (int)(im >> 16),
                                      (int)(im & 0xFFFF), lq, lt, ani, cov, filtered);
                    if (score_only) { rec.qb = rec.tb = 0; rec.ident = rec.cols = 0; rec.passes = 0; }
                    if (lane == 0) my_cells += (unsigned long long)lq * lt;
                }
                if (tune && lane == 0) atomicAdd(&tune[sw_bin(lq)], (unsigned long long)(clock64() - t_big));
            } else if (r1.score > 0 && (score_only || skip)) {
                rec.score = r1.score;                       // score and end only
                rec.qe = (uint16_t)(r1.end_i + 1);
                rec.te = (uint16_t)(r1.end_j + 1);
            } else if (r1.score > 0) {
                const int ri = r1.rect_i, rj = r1.rect_j;
                int h, dummy_i, dummy_j;
                uint32_t beg, im;
                // rows per lane from the rectangle's height, so that all 32 lanes have rows
                const int rows = r1.end_i + 1 - ri;
                const int ns3 = (rows + 32 * CR - 1) / (32 * CR);
                const int cr = min(CR, max(2, (((rows + 32 * ns3 - 1) / (32 * ns3)) + 1) & ~1));
                const uint8_t *cq = qcodes + qo + ri, *ct = tcodes + to + rj;
                const int cn = r1.end_j + 1 - rj;
#define PASTIS_CARRY_CASE(C) \
    case C: carry_warp<false, C>(cq, rows, ct, cn, s_mat, o, e, my, sstride, &h, &dummy_i, &dummy_j, &beg, &im); break;
                switch (cr) {
                    PASTIS_CARRY_CASE(2) PASTIS_CARRY_CASE(4) PASTIS_CARRY_CASE(6)
                    default: carry_warp<false, CR>(cq, rows, ct, cn, s_mat, o, e, my, sstride, &h, &dummy_i, &dummy_j,
                                                   &beg, &im); break;
                }
#undef PASTIS_CARRY_CASE
                if (h != r1.score && lane == 0) atomicExch(err, 1);
                finish_record(rec, r1.score, r1.end_i, r1.end_j, ri + (int)(beg >> 16), rj + (int)(beg & 0xFFFF),
                              (int)(im >> 16), (int)(im & 0xFFFF), lq, lt, ani, cov, filtered);
            }
            if (lane == 0) out[p] = rec;
        }
    }
    if (lane == 0 && cells && my_cells) atomicAdd(cells, my_cells);
}

}  // namespace

cudaError_t sw_set_smem_limit(size_t bytes) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, k_sw_score);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_sw_score, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(bytes - fa.sharedSizeBytes));
}

// Host side of the Smith-Waterman path (called by pastis_align_pairs after validation).
// dn != nullptr: a captured launch sequence (no host synchronisation): n_pairs is the
// capacity, the pair count is *dn in device memory, the row-pair bounds take their
// capacity bound, and chk (the input checks' flags) stops the kernels on bad input.
pastis_status sw_align(pastis_ctx *ctx, const uint8_t *d_qcodes, const int64_t *d_qoffsets, const uint8_t *d_tcodes,
                       const int64_t *d_toffsets, const pastis_cand *d_pairs,
                       int64_t n_pairs, const pastis_params *p, const int8_t *dmat, int *flags, int lmax,
                       pastis_aln *d_out, int64_t *d_cells, const int64_t *dn, const int *chk) {
    cudaStream_t st = ctx->stream;
    int max_s = 0;
    for (int x = 0; x < PASTIS_NSYM * PASTIS_NSYM; ++x) max_s = std::max(max_s, (int)p->matrix[x]);
    // segments of pairs sharing a query
    uint32_t *sflags;
    PASTIS_WS(sflags, ctx, WS_ALN_ORDER, sizeof(uint32_t) * (2 * (size_t)n_pairs + 2 + 2 * SEG_BINS) +
                                             sizeof(int64_t) * (n_pairs + 2) + 16);
    uint32_t *soff = sflags + n_pairs + 1, *hist = soff + n_pairs + 1;
    int64_t *seg_start = (int64_t *)(((uintptr_t)(hist + 2 * SEG_BINS) + 7) & ~(uintptr_t)7);
    PASTIS_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * 2 * SEG_BINS, st));
    k_seg_flags<<<(unsigned)ceil_div64(n_pairs, 256), 256, 0, st>>>(d_pairs, n_pairs, sflags, dn);
    PASTIS_LAUNCHED(ctx);
    pastis_status s = exclusive_scan_u32(ctx, sflags, soff, n_pairs);
    if (s != PASTIS_OK) return s;
    k_seg_starts<<<(unsigned)ceil_div64(n_pairs, 256), 256, 0, st>>>(d_pairs, d_qoffsets, sflags, soff, n_pairs,
                                                                     seg_start, hist, dn, chk);
    PASTIS_LAUNCHED(ctx);
    uint32_t h_nseg = 0;
    if (!dn) {
        PASTIS_CUDA_TRY(cudaMemcpyAsync(&h_nseg, soff + n_pairs, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
        PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    }

    // the flags have served: the segments' order takes their place
    const int64_t seg_cap = dn ? n_pairs : (int64_t)h_nseg;
    k_seg_order<<<(unsigned)ceil_div64(seg_cap, 256), 256, 0, st>>>(d_pairs, d_qoffsets, seg_start, seg_cap,
                                                                    dn ? soff + n_pairs : nullptr, hist,
                                                                    hist + SEG_BINS, sflags, chk);
    PASTIS_LAUNCHED(ctx);

    // row-pair bounds of pass 1 for pass 2: (query length + 1) / 2 int16 per pair
    int64_t *bm_cnt;
    PASTIS_WS(bm_cnt, ctx, WS_ALN_BOFF, sizeof(int64_t) * (2 * (size_t)n_pairs + 1));
    int64_t *bm_off = bm_cnt + n_pairs;
    k_bm_count<<<(unsigned)ceil_div64(n_pairs, 256), 256, 0, st>>>(d_pairs, n_pairs, d_qoffsets, bm_cnt, dn, chk);
    PASTIS_LAUNCHED(ctx);
    s = exclusive_scan_i64(ctx, bm_cnt, bm_off, n_pairs);
    if (s != PASTIS_OK) return s;
    int64_t h_bm = n_pairs * (int64_t)((lmax + 1) / 2);     // the bound of a captured sequence
    if (!dn) {
        PASTIS_CUDA_TRY(cudaMemcpyAsync(&h_bm, bm_off + n_pairs, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    }
    int16_t *bm_all;
    PASTIS_WS(bm_all, ctx, WS_ALN_BOUND, sizeof(int16_t) * (size_t)h_bm + 16);
    uint32_t *list = (uint32_t *)bm_cnt;       // the counts have served: two lists of pairs

    sw_score_out *res;
    PASTIS_WS(res, ctx, WS_ALN_PASS1, sizeof(sw_score_out) * (size_t)n_pairs);
    // pass 1+2: profile rows up to the longest query (in whole stripes), within shared memory
    int max_extra = 0;
    for (int b = 0; b < PASTIS_SW_BINS; ++b) max_extra = std::max(max_extra, (int)ctx->sw_lay.extra[b]);
    // profile bytes per residue: 512 up to 512 query rows, else 1,024 per 1,024 rows
    int prow_cap = lmax <= STRIPE1 && max_extra == 0 ? STRIPE1
                                                     : ((lmax + 2 * STRIPE1 - 1) / (2 * STRIPE1) + max_extra) * 2 * STRIPE1;
    auto shm_for = [](int pc) { return (size_t)NRES * pc; };
    while (prow_cap > STRIPE1 && shm_for(prow_cap) + 1088 > ctx->smem_optin) prow_cap -= STRIPE1;
    const size_t shm1 = shm_for(prow_cap);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sw_score, SW_THREADS, shm1);
    if (per_sm < 1) per_sm = 1;
    const int blocks1 = ctx->sm_count * per_sm;
    const int sstride = lmax + 1;
    const size_t warp_bytes = (sizeof(uint2) * 2 * (size_t)sstride + 255) & ~(size_t)255;
    const size_t scr1 = warp_bytes * (size_t)blocks1 * SW_WARPS;
    const int blocks3 = ctx->sm_count * 2;
    const size_t scr3 = sizeof(stripe3_cell) * (size_t)blocks3 * SW_WARPS * 2 * sstride;
    void *scratch;
    PASTIS_WS(scratch, ctx, WS_ALN_SCRATCH, std::max(scr1, scr3));
    // pass 2's column ranges per 8 rows; without room for them pass 3 takes the rectangles.
    // Taken last, so that they never have the room that a buffer needed above would take
    // (ws_get gives them up where a later call needs it).
    uint32_t *band = nullptr;
    if (p->mode != PASTIS_SW_SCORE) {
        const size_t bytes = sizeof(uint32_t) * ((size_t)(h_bm >> 2) + (size_t)n_pairs + 2);
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (dn) PASTIS_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
        // a capture allocates nothing: what its sizing run could not have, it goes without
        if (cap == cudaStreamCaptureStatusNone || ctx->ws_bytes[WS_ALN_BAND] >= bytes)
            band = (uint32_t *)ws_get(ctx, WS_ALN_BAND, bytes);
    }
    prof_begin(ctx, "sw_pass1");
    k_sw_score<<<blocks1, SW_THREADS, shm1, st>>>(d_qcodes, d_qoffsets, d_tcodes, d_toffsets, d_pairs, seg_start,
                                                  sflags, (int64_t)h_nseg, dmat,
                                                  p->gap_open, p->gap_extend, max_s, prow_cap, 1u, (char *)scratch,
                                                  warp_bytes, sstride, flags + 1, bm_all, bm_off, res,
                                                  (unsigned long long *)d_cells, (const uint8_t *)dmat + 640,
                                                  ctx->d_tune, dn ? soff + n_pairs : nullptr, chk);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    const int score_only = p->mode == PASTIS_SW_SCORE;
    const int filtered = p->mode == PASTIS_SW_FILTERED;
    int per_sm2 = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm2, k_sw_bound, SW_THREADS, 0);
    if (per_sm2 < 1) per_sm2 = 1;
    if (!score_only) {                         // the score mode needs no begin, so no rectangle
        prof_begin(ctx, "sw_pass2");
        k_sw_bound<<<ctx->sm_count * per_sm2, SW_THREADS, 0, st>>>(d_qcodes, d_qoffsets, d_tcodes, d_toffsets,
                                                                   d_pairs, n_pairs, dmat, p->gap_open, p->gap_extend,
                                                                   bm_all, bm_off, (unsigned long long *)(flags + 10),
                                                                   res, filtered ? p->cov_min_pct : -1, band, list,
                                                                   n_pairs, flags + 20, dn, chk);
        PASTIS_LAUNCHED(ctx);
        prof_end(ctx);
    }
    prof_begin(ctx, "sw_pass3");
    if (band) {
        const band_args g{d_qcodes, d_qoffsets, d_tcodes, d_toffsets, d_pairs, p->gap_open, p->gap_extend,
                          p->ani_min_pct, p->cov_min_pct, filtered, band, bm_off, list, n_pairs, flags + 20,
                          flags + 24, res, d_out, flags};
        k_sw_band<<<ctx->sm_count * 2, SW_THREADS, 0, st>>>(g, dmat, chk);
        PASTIS_LAUNCHED(ctx);
    }
    k_sw_carry<<<blocks3, SW_THREADS, 0, st>>>(d_qcodes, d_qoffsets, d_tcodes, d_toffsets, d_pairs, n_pairs, dmat,
                                               p->gap_open,
                                               p->gap_extend, p->ani_min_pct, p->cov_min_pct,
                                               (stripe3_cell *)scratch, sstride, flags + 8, res, score_only, filtered,
                                               d_out, flags,
                                               (unsigned long long *)d_cells, ctx->d_tune, dn, chk);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    return PASTIS_OK;
}
