// a4-a5: substitute k-mers (the matrix S) and the product AS.
//
// Sec. IV-B: the expense of replacing base a by b is C[a][a] - C[a][b] (the matrix
// E = Sort(Diag(C) - C)); a k-mer's distance from a root is the sum of its per-position
// expenses.  Row r of S holds r itself (distance 0) and the m k-mers q != r nearest to
// r, ties broken by the smaller code.  Alg. 1-3 reach that set with a best-first
// search over min-max heaps; on the GPU each thread owns one root and finds it in two
// fixed-size phases instead:
//   1. the number of k-mers at every distance, as a convolution over positions of the
//      per-position expense histograms; it yields the cut distance D* (the first
//      distance at which at least m k-mers q != r are reached) and how many of the
//      ties at D* are taken;
//   2. one depth-first walk of the k-mer tree in code order, pruned at D*: every
//      k-mer closer than D* and the first `quota` ones at D* are written straight to
//      their sorted slot, slot = (number of k-mers closer than it) + (its rank among
//      equal distances in code order).
// Sec. IV-C: AS(i, s) keeps the start of the k-mer of sequence i nearest to s (the
// smaller start on ties).  Both products meet AS only at codes that A holds (AS rows against
// A's posting lists, A's rows against AS's), so only the substitutes present in A are
// kept: about a seventh of them at 20,000 proteins (182 M entries; building AS and the product
// 31 ms with all of them, 12 ms so), two fifths at 100,000.  AS is expanded from the
// rows of A and these rows of S, radix-sorted by s (stable, so sequences stay ascending),
// reduced to one entry per (s, i), and sorted again by sequence for its CSR view.
#include <string.h>

#include "internal.cuh"

namespace {

constexpr int SUBK_DLIM = 64;     // shifted distances handled (see check_params bounds)
constexpr int SUBK_NEAR = 16;     // shifted distances counted in registers first
constexpr int SUBK_THREADS = 128;

// Phase 1: the number of k-mers at each shifted distance, one position at a time (counts
// of the prefixes convolved with the residue's expense histogram); then the cut (-1:
// fewer than m k-mers q != r are closer than the distances counted), the number closer
// than it (*below), and the slot of the first k-mer of each distance (base).  Here over
// the first 16 distances, in registers, 16 byte counts a load.
__device__ __forceinline__ int subk_cut_near(const uint8_t *s_hist, uint32_t digs, int k, int m, int xr,
                                             uint8_t *base, int bstride, int *below) {
    int cnt[SUBK_NEAR];
#pragma unroll
    for (int x = 0; x < SUBK_NEAR; ++x) cnt[x] = x == 0;
    for (int t = 0; t < k; ++t) {
        const uint4 w = *reinterpret_cast<const uint4 *>(s_hist + ((digs >> (5 * t)) & 31u) * SUBK_DLIM);
        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
        int nw[SUBK_NEAR];
#pragma unroll
        for (int x = 0; x < SUBK_NEAR; ++x) nw[x] = 0;
#pragma unroll
        for (int s = 0; s < SUBK_NEAR; ++s) {
            const int h = (int)((ws[s >> 2] >> (8 * (s & 3))) & 0xFFu);
#pragma unroll
            for (int x = s; x < SUBK_NEAR; ++x) nw[x] += h * cnt[x - s];
        }
#pragma unroll
        for (int x = 0; x < SUBK_NEAR; ++x) cnt[x] = nw[x];
    }
    int cut = -1, run = 0;
#pragma unroll
    for (int x = 0; x < SUBK_NEAR; ++x) {
        const int here = cnt[x] - (x == xr ? 1 : 0);
        if (cut < 0) {
            base[x * bstride] = (uint8_t)run;          // run < m <= 128
            if (run + here >= m) { cut = x; *below = run; }
        }
        run += here;
    }
    return cut;
}

// The same over all SUBK_DLIM distances, for the roots whose cut lies further out.
__device__ __noinline__ int subk_cut_far(const uint8_t *s_hist, uint32_t digs, int k, int m, int xr, uint8_t *base,
                                         int bstride, int *below) {
    int cnt[SUBK_DLIM];
#pragma unroll 1
    for (int x = 0; x < SUBK_DLIM; ++x) cnt[x] = x == 0;
#pragma unroll 1
    for (int t = 0; t < k; ++t) {
        const uint8_t *h = s_hist + ((digs >> (5 * t)) & 31u) * SUBK_DLIM;
#pragma unroll 1
        for (int x = SUBK_DLIM - 1; x >= 0; --x) {     // in place: position x reads only x and below
            int v = 0;
#pragma unroll 1
            for (int s = 0; s <= x; ++s) v += (int)h[s] * cnt[x - s];
            cnt[x] = v;
        }
    }
    int run = 0;
#pragma unroll 1
    for (int x = 0; x < SUBK_DLIM; ++x) {
        const int here = cnt[x] - (x == xr ? 1 : 0);
        base[x * bstride] = (uint8_t)run;
        if (run + here >= m) { *below = run; return x; }
        run += here;
    }
    return -1;
}

// One thread per root: about 700 multiply-adds of phase 1 (16 distances hold the cut of
// nearly every root with BLOSUM62; the others are counted again over all 64) and a dozen
// instructions for each step of the walk.  What bounds it is the walks' divergence: 12.5 of 32
// lanes are active in an instruction and the issue slots are two thirds busy; the rest is
// branches and dependent steps that 18 warps an SM (their rows in shared memory) do not
// hide.  A bit
// mask per (residue, budget) names the replacements that keep a prefix within the cut,
// so the walk touches only prefixes that lead to a k-mer it keeps or a tie at the cut;
// its stack, the running slot of each distance and the rows under construction live in
// shared memory, and a CTA's rows, contiguous in the output, leave in one linear copy.
// Measured with m = 25 and k = 6 on the distinct 6-mers of 20,000 proteins: 69.8 ms with the
// counts in local memory and every replacement tried at every level, 6.0 ms so.
// PRESENT: only the entries whose code's bit is set in `bits` leave, in their order at the
// front of the root's row, and their number in out_n.
template <bool PRESENT>
__global__ void __launch_bounds__(SUBK_THREADS) k_subkmers(const uint32_t *__restrict__ roots, int64_t n_roots,
                                                           int k, int m, const int8_t *__restrict__ gmat,
                                                           const uint32_t *__restrict__ bits,
                                                           uint32_t *__restrict__ out_code,
                                                           int32_t *__restrict__ out_dist,
                                                           uint32_t *__restrict__ out_n, int *err) {
    extern __shared__ __align__(16) unsigned char subk_smem[];
    __shared__ __align__(16) uint8_t s_hist[PASTIS_NSYM * SUBK_DLIM];   // replacements of a residue at each expense
    __shared__ uint32_t s_mask[PASTIS_NSYM * SUBK_DLIM];                // replacements of a residue within a budget
    __shared__ uint8_t s_exp[PASTIS_NSYM * PASTIS_NSYM];                // shifted expenses (0..254)
    __shared__ int s_min[PASTIS_NSYM];
    const int T = blockDim.x, tid = threadIdx.x;
    uint32_t *s_code = reinterpret_cast<uint32_t *>(subk_smem);         // [T][m + 1]
    uint32_t *s_stm = s_code + T * (m + 1);                             // [5][T] masks left on the levels above
    uint32_t *s_stp = s_stm + 5 * T;                                    // [5][T] their prefixes
    int16_t *s_dist = reinterpret_cast<int16_t *>(s_stp + 5 * T);       // [T][m + 1]
    uint8_t *s_base = reinterpret_cast<uint8_t *>(s_dist + T * (m + 1));  // [64][T]
    if (tid < PASTIS_NSYM) {
        const int own = gmat[tid * PASTIS_NSYM + tid];
        int mn = own - (int)gmat[tid * PASTIS_NSYM];
        for (int b = 1; b < PASTIS_NSYM; ++b) mn = min(mn, own - (int)gmat[tid * PASTIS_NSYM + b]);
        s_min[tid] = mn;
        for (int b = 0; b < PASTIS_NSYM; ++b)
            s_exp[tid * PASTIS_NSYM + b] = (uint8_t)(own - (int)gmat[tid * PASTIS_NSYM + b] - mn);
        for (int d = 0; d < SUBK_DLIM; ++d) {
            int h = 0;
            uint32_t w = 0;
            for (int b = 0; b < PASTIS_NSYM; ++b) {
                const int x = s_exp[tid * PASTIS_NSYM + b];
                h += x == d;
                w |= x <= d ? 1u << b : 0u;
            }
            s_hist[tid * SUBK_DLIM + d] = (uint8_t)h;
            s_mask[tid * SUBK_DLIM + d] = w;
        }
    }
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * T;
    const int64_t r = r0 + tid;
    if (r < n_roots) {
        const uint32_t root = roots[r];
        uint32_t digs = 0;             // 5 bits per position, position 0 lowest
        int shift_total = 0;           // sum of per-position minima (unshifted = shifted + shift_total)
        uint32_t x = root;
        for (int t = k - 1; t >= 0; --t) {
            const uint32_t d = x % PASTIS_NSYM;
            x /= PASTIS_NSYM;
            digs |= d << (5 * t);
            shift_total += s_min[d];
        }
        uint32_t *code_row = s_code + tid * (m + 1);
        int16_t *dist_row = s_dist + tid * (m + 1);
        code_row[0] = root;
        dist_row[0] = 0;
        uint8_t *base = s_base + tid;
        const int xr = -shift_total;   // shifted distance of the root itself
        int below = 0;
        int cut = m == 0 ? -1 : subk_cut_near(s_hist, digs, k, m, xr, base, T, &below);
        if (m > 0 && cut < 0) {
            cut = subk_cut_far(s_hist, digs, k, m, xr, base, T, &below);
            if (cut < 0) atomicExch(err, 1);
        }
        if (cut >= 0) {
            int quota = m - below;
            // phase 2: depth-first walk in code order, pruned at the cut.  A prefix is one
            // word: its code (below 24^5), its distance and whether it is the root's.
            int depth = 0;
            uint32_t pc = 1u << 31;
            uint32_t mask = s_mask[(digs & 31u) * SUBK_DLIM + cut];
            for (;;) {
                if (mask == 0u) {
                    if (depth == 0) break;
                    --depth;
                    mask = s_stm[depth * T + tid];
                    pc = s_stp[depth * T + tid];
                    continue;
                }
                const uint32_t b = (uint32_t)__ffs(mask) - 1u;
                mask &= mask - 1u;
                const uint32_t d = (digs >> (5 * depth)) & 31u;
                const uint32_t ps = ((pc >> 24) & 63u) + s_exp[d * PASTIS_NSYM + b];
                const uint32_t code = (pc & 0xFFFFFFu) * PASTIS_NSYM + b;
                const bool is_root = (pc >> 31) && b == d;
                if (depth + 1 < k) {
                    s_stm[depth * T + tid] = mask;
                    s_stp[depth * T + tid] = pc;
                    ++depth;
                    pc = (is_root ? 1u << 31 : 0u) | (ps << 24) | code;
                    mask = s_mask[((digs >> (5 * depth)) & 31u) * SUBK_DLIM + (cut - (int)ps)];
                    continue;
                }
                if (is_root) continue;
                if ((int)ps == cut) {
                    if (quota == 0) continue;
                    --quota;
                }
                const int slot = base[ps * T]++;
                code_row[1 + slot] = code;
                dist_row[1 + slot] = (int16_t)((int)ps + shift_total);
            }
        }
        if (PRESENT) {
            uint32_t cnt = 0;
            const int64_t o = r * (m + 1);
            for (int w0 = 0; w0 <= m && (cut >= 0 || m == 0); w0 += 8) {
                uint32_t word[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) word[u] = w0 + u <= m ? bits[code_row[w0 + u] >> 5] : 0u;
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (w0 + u > m) break;
                    const uint32_t code = code_row[w0 + u];
                    if ((word[u] >> (code & 31u)) & 1u) {
                        out_code[o + cnt] = code;
                        out_dist[o + cnt] = dist_row[w0 + u];
                        ++cnt;
                    }
                }
            }
            out_n[r] = cnt;
        }
    }
    if (PRESENT) return;
    __syncthreads();
    const int64_t left = n_roots - r0;
    const int words = (int)(left < T ? left : T) * (m + 1);
    uint32_t *oc = out_code + r0 * (m + 1);
    int32_t *od = out_dist + r0 * (m + 1);
    for (int w = tid; w < words; w += T) {
        oc[w] = s_code[w];
        od[w] = s_dist[w];
    }
}

// Shared memory of a CTA of T threads, and the widest CTA whose rows leave several CTAs
// on an SM: 128 threads up to m = 33, 32 at m = 128.
size_t subk_smem_bytes(int T, int m) { return (size_t)T * ((m + 1) * 6 + 40 + SUBK_DLIM); }
int subk_threads(int m) {
    int T = SUBK_THREADS;
    while (T > 32 && subk_smem_bytes(T, m) > (39u << 10)) T >>= 1;
    return T;
}

// The codes A holds, as a bit map over all codes (one read of col_ptr), with the number set
// in each tile of ROOT_TILE codes.
constexpr int ROOT_THREADS = 256, ROOT_TILE = ROOT_THREADS * 32;

__global__ void __launch_bounds__(ROOT_THREADS) k_present_bits(const uint32_t *__restrict__ col_ptr, int64_t ncodes,
                                                               uint32_t *__restrict__ bits,
                                                               uint32_t *__restrict__ tile_n) {
    __shared__ uint32_t s_n[ROOT_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t c0 = (int64_t)blockIdx.x * ROOT_TILE;
    uint32_t n = 0;
#pragma unroll 4
    for (int w = warp; w < ROOT_TILE / 32; w += ROOT_THREADS / 32) {
        const int64_t c = c0 + w * 32 + lane;
        const uint32_t here = c <= ncodes ? col_ptr[c] : 0u;
        uint32_t next = __shfl_down_sync(0xffffffffu, here, 1);
        if (lane == 31) next = c < ncodes ? col_ptr[c + 1] : 0u;
        const uint32_t b = __ballot_sync(0xffffffffu, c < ncodes && next > here);
        if (lane == 0 && c0 + w * 32 < ncodes) bits[(c0 >> 5) + w] = b;
        n += __popc(b);
    }
    if (lane == 0) s_n[warp] = n;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < ROOT_THREADS / 32; ++w) t += s_n[w];
        tile_n[blockIdx.x] = t;
    }
}

// The present codes in order, and before each word of the bit map the number set before it,
// so that a code's place among the roots is two cached reads.
__global__ void __launch_bounds__(ROOT_THREADS) k_roots(const uint32_t *__restrict__ bits, int64_t nwords,
                                                        const uint32_t *__restrict__ tile_off,
                                                        uint32_t *__restrict__ before, uint32_t *__restrict__ roots) {
    __shared__ uint32_t s_n[ROOT_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w = (int64_t)blockIdx.x * ROOT_THREADS + threadIdx.x;
    uint32_t b = w < nwords ? bits[w] : 0u;
    uint32_t incl = __popc(b);
    const uint32_t own = incl;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    if (lane == 31) s_n[warp] = incl;
    __syncthreads();
    uint32_t at = tile_off[blockIdx.x] + incl - own;
    for (int u = 0; u < warp; ++u) at += s_n[u];
    if (w < nwords) before[w] = at;
    while (b) {
        const int x = __ffs(b) - 1;
        b &= b - 1u;
        roots[at++] = (uint32_t)(w * 32 + x);
    }
}

__device__ __forceinline__ uint32_t root_of(const uint32_t *bits, const uint32_t *before, uint32_t code) {
    const uint32_t w = code >> 5;
    return before[w] + __popc(bits[w] & ((1u << (code & 31u)) - 1u));
}

// Substitutes kept for each entry of A.
__global__ void k_as_count(const uint32_t *__restrict__ row_code, int64_t nnz, const uint32_t *__restrict__ bits,
                           const uint32_t *__restrict__ before, const uint32_t *__restrict__ sub_n,
                           uint32_t *__restrict__ cnt) {
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x < nnz) cnt[x] = sub_n[root_of(bits, before, row_code[x])];
}

// Expansion of AS: entry x of A row i and substitute t of its code becomes key =
// substitute code, value = i << 32 | dist << 16 | pos, from off[x] on.  Rows are walked in
// order, so equal substitutes keep ascending i after a stable sort by key.
__global__ void __launch_bounds__(256) k_expand_as(const int64_t *__restrict__ row_ptr,
                                                   const uint32_t *__restrict__ row_code,
                                                   const uint16_t *__restrict__ row_pos, int32_t n, int64_t nnz,
                                                   const uint32_t *__restrict__ bits,
                                                   const uint32_t *__restrict__ before,
                                                   const uint32_t *__restrict__ sub_code,
                                                   const int32_t *__restrict__ sub_dist, int m,
                                                   const uint32_t *__restrict__ off, uint32_t *__restrict__ keys,
                                                   uint64_t *__restrict__ vals) {
    // the rows of the CTA's first and last entry bound the search of each
    __shared__ int32_t s_row[2];
    const int64_t x0 = (int64_t)blockIdx.x * blockDim.x, x = x0 + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < 2) {
        const int64_t y = warp == 0 ? x0 : min(x0 + blockDim.x, nnz) - 1;
        int64_t lo = 0, hi = n - 1;              // the last row with row_ptr[row] <= y
        while (lo < hi) {
            const int64_t step = (hi - lo + 31) / 32, r = lo + step * (lane + 1);
            const int c = __popc(__ballot_sync(0xffffffffu, r <= hi && row_ptr[r] <= y));
            const int64_t nlo = lo + step * c;
            hi = min(hi, nlo + step - 1);
            lo = nlo;
        }
        if (lane == 0) s_row[warp] = (int32_t)lo;
    }
    __syncthreads();
    if (x >= nnz) return;
    int32_t lo = s_row[0], hi = s_row[1];
    while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (row_ptr[mid] <= x) lo = mid; else hi = mid - 1;
    }
    const int64_t sidx = (int64_t)root_of(bits, before, row_code[x]) * (m + 1);
    const uint64_t base = ((uint64_t)(uint32_t)lo << 32) | row_pos[x];
    const uint32_t o = off[x], c = off[x + 1] - o;
    for (uint32_t t = 0; t < c; ++t) {
        keys[o + t] = sub_code[sidx + t];
        // distances are biased by 1024 so that (dist, pos) orders as one unsigned word
        vals[o + t] = base | ((uint64_t)(uint32_t)(sub_dist[sidx + t] + 1024) << 16);
    }
}

// After the sort by substitute code: the first entry of each (code, seq) run becomes the
// run's minimum (dist, pos) and is flagged to keep.
__global__ void k_reduce_as_runs(const uint32_t *keys, uint64_t *vals, int64_t n, uint32_t *keep) {
    int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    uint32_t key = keys[x];
    uint64_t v = vals[x];
    uint32_t seq = (uint32_t)(v >> 32);
    if (x > 0 && keys[x - 1] == key && (uint32_t)(vals[x - 1] >> 32) == seq) { keep[x] = 0; return; }
    uint32_t best = (uint32_t)(v & 0xFFFFFFFFu);   // dist << 16 | pos, both non-negative
    for (int64_t y = x + 1; y < n && keys[y] == key && (uint32_t)(vals[y] >> 32) == seq; ++y) {
        uint32_t w = (uint32_t)(vals[y] & 0xFFFFFFFFu);
        if (w < best) best = w;
    }
    vals[x] = ((uint64_t)seq << 32) | best;
    keep[x] = 1;
}

__global__ void k_compact_as(const uint32_t *keys, const uint64_t *vals, const uint32_t *keep,
                             const uint32_t *off, int64_t n, int32_t *col_seq, uint16_t *col_pos,
                             uint32_t *rkeys, uint64_t *rvals) {
    int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n || !keep[x]) return;
    uint32_t o = off[x];
    uint32_t seq = (uint32_t)(vals[x] >> 32);
    uint16_t pos = (uint16_t)(vals[x] & 0xFFFF);
    col_seq[o] = (int32_t)seq;
    col_pos[o] = pos;
    rkeys[o] = seq;
    rvals[o] = ((uint64_t)keys[x] << 16) | pos;
}

// row_ptr[r] = first index x with keys[x] >= r (keys sorted ascending), r = 0..n
__global__ void k_row_count_u32(const uint32_t *keys, int64_t nnz, int32_t n, int64_t *row_ptr) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r > n) return;
    int64_t lo = 0, hi = nnz;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if ((int64_t)keys[mid] < r) lo = mid + 1; else hi = mid;
    }
    row_ptr[r] = lo;
}

__global__ void k_split_rows_as(const uint64_t *rvals, int64_t nnz, uint32_t *row_code, uint16_t *row_pos) {
    int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nnz) return;
    row_code[x] = (uint32_t)(rvals[x] >> 16);
    row_pos[x] = (uint16_t)(rvals[x] & 0xFFFF);
}

int bits_for_u64(uint64_t v) {
    int b = 0;
    while (b < 64 && (v >> b) != 0) ++b;
    return b;
}

pastis_status launch_subkmers(pastis_ctx *ctx, const uint32_t *d_roots, int64_t n_roots, int k, int m,
                              const pastis_params *params, uint32_t *d_code, int32_t *d_dist,
                              const uint32_t *d_bits = nullptr, uint32_t *d_n = nullptr) {
    int8_t *dmat;
    PASTIS_WS(dmat, ctx, WS_FLAGS, 1024);
    int *err = (int *)(dmat + 768);
    PASTIS_CUDA_TRY(cudaMemcpyAsync(dmat, params->matrix, 576, cudaMemcpyHostToDevice, ctx->stream));
    PASTIS_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), ctx->stream));
    if (n_roots > 0) {
        prof_begin(ctx, "subkmers");
        const int T = subk_threads(m);
        auto kern = d_bits ? k_subkmers<true> : k_subkmers<false>;
        kern<<<(unsigned)ceil_div64(n_roots, T), T, subk_smem_bytes(T, m), ctx->stream>>>(
            d_roots, n_roots, k, m, dmat, d_bits, d_code, d_dist, d_n, err);
        PASTIS_LAUNCHED(ctx);
        prof_end(ctx);
    }
    int herr = 0;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    PASTIS_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    return herr ? PASTIS_ERR_INTERNAL : PASTIS_OK;
}

}  // namespace

extern "C" pastis_status pastis_substitute_kmers(pastis_ctx *ctx, const uint32_t *d_roots, int64_t n_roots,
                                                 const pastis_params *params, uint32_t *d_sub_code,
                                                 int32_t *d_sub_dist) {
    if (!ctx || n_roots < 0 || (n_roots > 0 && (!d_roots || !d_sub_code || !d_sub_dist)))
        return PASTIS_ERR_INVALID_ARG;
    pastis_status s = check_params(params);
    if (s != PASTIS_OK) return s;
    return launch_subkmers(ctx, d_roots, n_roots, params->k, params->m_subs, params, d_sub_code, d_sub_dist);
}

// Sets *flag when a[x] != b[x] for some x < n.
template <typename T>
__global__ void k_differs(const T *__restrict__ a, const T *__restrict__ b, int64_t n, uint32_t *flag) {
    bool d = false;
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x)
        d |= a[x] != b[x];
    if (__any_sync(0xffffffffu, d) && (threadIdx.x & 31) == 0) atomicOr(flag, 1u);
}

// Layout of the kept copy of A's rows: the flag word, then row_ptr, row_code, row_pos.
struct as_keep_view {
    uint32_t *flag;
    int64_t *row_ptr;
    uint32_t *row_code;
    uint16_t *row_pos;
};
static size_t as_keep_bytes(int64_t n, int64_t nnz) {
    return 256 + sizeof(int64_t) * (size_t)(n + 1) + sizeof(uint32_t) * (size_t)nnz + sizeof(uint16_t) * (size_t)nnz + 64;
}
static as_keep_view as_keep_layout(void *base, int64_t n, int64_t nnz) {
    as_keep_view v;
    char *p = (char *)base;
    v.flag = (uint32_t *)p;
    v.row_ptr = (int64_t *)(p + 256);
    v.row_code = (uint32_t *)(v.row_ptr + n + 1);
    v.row_pos = (uint16_t *)(v.row_code + nnz);
    return v;
}

// True when the kept AS was built from this A (same rows, compared on the device), k,
// m and matrix.  Synchronises the stream.
static pastis_status as_kept_matches(pastis_ctx *ctx, const pastis_kmat *A, const pastis_params *p, bool *hit) {
    *hit = false;
    if (!ctx->as_valid || ctx->as_k != p->k || ctx->as_m != p->m_subs || ctx->as_n != A->n_rows ||
        ctx->as_nnz_a != A->nnz || memcmp(ctx->as_mat, p->matrix, sizeof(ctx->as_mat)) != 0)
        return PASTIS_OK;
    cudaStream_t st = ctx->stream;
    const as_keep_view v = as_keep_layout(ctx->ws[WS_AS_KEEP], A->n_rows, A->nnz);
    PASTIS_CUDA_TRY(cudaMemsetAsync(v.flag, 0, sizeof(uint32_t), st));
    const int blocks = ctx->sm_count * 8;
    k_differs<int64_t><<<blocks, 256, 0, st>>>(A->row_ptr, v.row_ptr, (int64_t)A->n_rows + 1, v.flag);
    PASTIS_LAUNCHED(ctx);
    if (A->nnz > 0) {
        k_differs<uint32_t><<<blocks, 256, 0, st>>>(A->row_code, v.row_code, A->nnz, v.flag);
        PASTIS_LAUNCHED(ctx);
        k_differs<uint16_t><<<blocks, 256, 0, st>>>(A->row_pos, v.row_pos, A->nnz, v.flag);
        PASTIS_LAUNCHED(ctx);
    }
    uint32_t h = 1;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(&h, v.flag, sizeof(h), cudaMemcpyDeviceToHost, st));
    PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    *hit = h == 0;
    return PASTIS_OK;
}

// Keeps a copy of A's rows beside the AS just built, so that a later product over the
// same A (another row block) reuses it.
static pastis_status as_keep(pastis_ctx *ctx, const pastis_kmat *A, const pastis_params *p, const as_matrix *AS) {
    void *base;
    PASTIS_WS(base, ctx, WS_AS_KEEP, as_keep_bytes(A->n_rows, A->nnz));
    const as_keep_view v = as_keep_layout(base, A->n_rows, A->nnz);
    cudaStream_t st = ctx->stream;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(v.row_ptr, A->row_ptr, sizeof(int64_t) * ((size_t)A->n_rows + 1),
                                    cudaMemcpyDeviceToDevice, st));
    if (A->nnz > 0) {
        PASTIS_CUDA_TRY(cudaMemcpyAsync(v.row_code, A->row_code, sizeof(uint32_t) * (size_t)A->nnz,
                                        cudaMemcpyDeviceToDevice, st));
        PASTIS_CUDA_TRY(cudaMemcpyAsync(v.row_pos, A->row_pos, sizeof(uint16_t) * (size_t)A->nnz,
                                        cudaMemcpyDeviceToDevice, st));
    }
    ctx->as_k = p->k;
    ctx->as_m = p->m_subs;
    ctx->as_n = A->n_rows;
    ctx->as_nnz_a = A->nnz;
    memcpy(ctx->as_mat, p->matrix, sizeof(ctx->as_mat));
    ctx->as_kept = *AS;
    ctx->as_valid = 1;
    return PASTIS_OK;
}

// Builds AS (Sec. IV-C), or reuses the one kept from the last call when A, k, m and the
// matrix are unchanged: S depends only on the k-mers present and AS only on A and S, so
// the row blocks of one job share them.
pastis_status build_as_fresh(pastis_ctx *ctx, const pastis_kmat *A, const pastis_params *p, as_matrix *out);

pastis_status build_as(pastis_ctx *ctx, const pastis_kmat *A, const pastis_params *p, as_matrix *out) {
    bool hit = false;
    pastis_status s = as_kept_matches(ctx, A, p, &hit);
    if (s != PASTIS_OK) return s;
    if (hit) {
        *out = ctx->as_kept;
        return PASTIS_OK;
    }
    ctx->as_valid = 0;
    s = build_as_fresh(ctx, A, p, out);
    if (s != PASTIS_OK) return s;
    return as_keep(ctx, A, p, out);
}

pastis_status build_as_fresh(pastis_ctx *ctx, const pastis_kmat *A, const pastis_params *p, as_matrix *out) {
    cudaStream_t st = ctx->stream;
    const int k = p->k, m = p->m_subs;
    const int64_t ncodes = ipow24(k);
    const int32_t n = A->n_rows;
    const int64_t nnzA = A->nnz;
    // the products of rows and substitutes that fit the sort's indexes
    if (nnzA * (m + 1) > 0xFFFFFFFFll) return PASTIS_ERR_UNSUPPORTED;
    // the codes present in A: bit map, rank, and the roots in order
    const int64_t nwords = ceil_div64(ncodes, 32), ntile = ceil_div64(ncodes, ROOT_TILE);
    uint32_t *bits;
    PASTIS_WS(bits, ctx, WS_SUB_ROOTS, sizeof(uint32_t) * (2 * (size_t)nwords + 2 * (size_t)ntile + 2));
    uint32_t *before = bits + nwords, *tile_n = before + nwords, *tile_off = tile_n + ntile;
    prof_begin(ctx, "as_roots");
    k_present_bits<<<(unsigned)ntile, ROOT_THREADS, 0, st>>>(A->col_ptr, ncodes, bits, tile_n);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    pastis_status s = exclusive_scan_u32(ctx, tile_n, tile_off, ntile);
    if (s != PASTIS_OK) return s;
    uint32_t h_nroots = 0;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(&h_nroots, tile_off + ntile, 4, cudaMemcpyDeviceToHost, st));
    PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    const int64_t nroots = h_nroots;
    uint32_t *roots, *sc;
    int32_t *sd;
    PASTIS_WS(roots, ctx, WS_AS_TMP_KEY, 2 * sizeof(uint32_t) * (nroots + 1));
    uint32_t *sub_n = roots + nroots + 1;
    PASTIS_WS(sc, ctx, WS_SUB_CODE, sizeof(uint32_t) * (nroots + 1) * (m + 1));
    PASTIS_WS(sd, ctx, WS_SUB_DIST, sizeof(int32_t) * (nroots + 1) * (m + 1));
    k_roots<<<(unsigned)ntile, ROOT_THREADS, 0, st>>>(bits, nwords, tile_off, before, roots);
    PASTIS_LAUNCHED(ctx);
    s = launch_subkmers(ctx, roots, nroots, k, m, p, sc, sd, bits, sub_n);
    if (s != PASTIS_OK) return s;
    // expand AS: the kept substitutes of every entry of A
    uint32_t *cnt;
    PASTIS_WS(cnt, ctx, WS_KMER_TMP, sizeof(uint32_t) * (2 * (size_t)nnzA + 2));
    uint32_t *cnt_off = cnt + nnzA + 1;
    if (nnzA > 0) {
        k_as_count<<<(unsigned)ceil_div64(nnzA, 256), 256, 0, st>>>(A->row_code, nnzA, bits, before, sub_n, cnt);
        PASTIS_LAUNCHED(ctx);
    }
    s = exclusive_scan_u32(ctx, cnt, cnt_off, nnzA);
    if (s != PASTIS_OK) return s;
    uint32_t h_ne = 0;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(&h_ne, cnt_off + nnzA, 4, cudaMemcpyDeviceToHost, st));
    PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    const int64_t ne = h_ne;
    uint32_t *ka, *kb;
    uint64_t *va, *vb;
    PASTIS_WS(ka, ctx, WS_SORT_KEYS_A, sizeof(uint32_t) * (ne + 1));
    PASTIS_WS(kb, ctx, WS_SORT_KEYS_B, sizeof(uint32_t) * (ne + 1));
    PASTIS_WS(va, ctx, WS_SORT_VALS_A, sizeof(uint64_t) * (ne + 1));
    PASTIS_WS(vb, ctx, WS_SORT_VALS_B, sizeof(uint64_t) * (ne + 1));
    if (ne > 0) {
        prof_begin(ctx, "as_expand");
        k_expand_as<<<(unsigned)ceil_div64(nnzA, 256), 256, 0, st>>>(A->row_ptr, A->row_code, A->row_pos, n, nnzA, bits,
                                                                     before, sc, sd, m, cnt_off, ka, va);
        PASTIS_LAUNCHED(ctx);
        prof_end(ctx);
    }
    uint32_t *sk;
    uint64_t *sv;
    s = radix_sort_u32_u64(ctx, ka, va, kb, vb, ne, bits_for_u64((uint64_t)ncodes), &sk, &sv);
    if (s != PASTIS_OK) return s;
    uint32_t *keep;
    PASTIS_WS(keep, ctx, WS_KMER_TMP, sizeof(uint32_t) * (2 * (size_t)ne + 2));
    uint32_t *off = keep + ne + 1;
    if (ne > 0) {
        prof_begin(ctx, "as_reduce");
        k_reduce_as_runs<<<(unsigned)ceil_div64(ne, 256), 256, 0, st>>>(sk, sv, ne, keep);
        PASTIS_LAUNCHED(ctx);
        prof_end(ctx);
    }
    s = exclusive_scan_u32(ctx, keep, off, ne);
    if (s != PASTIS_OK) return s;
    uint32_t h_nnz = 0;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(&h_nnz, off + ne, 4, cudaMemcpyDeviceToHost, st));
    PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    const int64_t nnz = h_nnz;
    out->nnz = nnz;
    PASTIS_WS(out->col_ptr, ctx, WS_AS_COLPTR, sizeof(uint32_t) * (ncodes + 1));
    PASTIS_WS(out->col_seq, ctx, WS_AS_COLSEQ, sizeof(int32_t) * (nnz + 1));
    PASTIS_WS(out->col_pos, ctx, WS_AS_COLPOS, sizeof(uint16_t) * (nnz + 1));
    PASTIS_WS(out->row_ptr, ctx, WS_AS_ROWPTR, sizeof(int64_t) * (n + 1));
    PASTIS_WS(out->row_code, ctx, WS_AS_CODE, sizeof(uint32_t) * (nnz + 1));
    PASTIS_WS(out->row_pos, ctx, WS_AS_POS, sizeof(uint16_t) * (nnz + 1));
    uint32_t *rk = (sk == ka) ? kb : ka;
    uint64_t *rv = (sv == va) ? vb : va;
    if (ne > 0) {
        prof_begin(ctx, "as_compact");
        k_compact_as<<<(unsigned)ceil_div64(ne, 256), 256, 0, st>>>(sk, sv, keep, off, ne, out->col_seq,
                                                                   out->col_pos, rk, rv);
        PASTIS_LAUNCHED(ctx);
        prof_end(ctx);
    }
    s = fill_col_ptr(ctx, sk, off, ne, ncodes, out->col_ptr);
    if (s != PASTIS_OK) return s;
    uint32_t *rko;
    uint64_t *rvo;
    s = radix_sort_u32_u64(ctx, rk, rv, sk, sv, nnz, bits_for_u64((uint64_t)(n > 0 ? n - 1 : 0)), &rko, &rvo);
    if (s != PASTIS_OK) return s;
    prof_begin(ctx, "as_rowptr");
    k_row_count_u32<<<(unsigned)ceil_div64((int64_t)n + 1, 256), 256, 0, st>>>(rko, nnz, n, out->row_ptr);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    if (nnz > 0) {
        k_split_rows_as<<<(unsigned)ceil_div64(nnz, 256), 256, 0, st>>>(rvo, nnz, out->row_code, out->row_pos);
        PASTIS_LAUNCHED(ctx);
    }
    return PASTIS_OK;
}
