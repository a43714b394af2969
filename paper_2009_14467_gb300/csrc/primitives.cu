// Device primitives used by the k-mer and candidate stages: a reduce-then-scan exclusive
// prefix sum and a stable LSD radix sort (digits of 5 to 8 bits) of (uint32 key, uint64 value).
#include "internal.cuh"

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
__device__ T block_exclusive_scan(T v, T *s_warp, T *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < (SCAN_THREADS / 32) ? s_warp[lane] : T(0);
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, w, d);
            if (lane >= d) w += y;
        }
        if (lane < (SCAN_THREADS / 32)) s_warp[lane] = w;
    }
    __syncthreads();
    T warp_off = warp > 0 ? s_warp[warp - 1] : T(0);
    *total = s_warp[SCAN_THREADS / 32 - 1];
    __syncthreads();
    return warp_off + x - v;
}

template <typename TI, typename TO>
__global__ void __launch_bounds__(SCAN_THREADS) k_tile_reduce(const TI *in, int64_t n, TO *sums) {
    __shared__ TO s_warp[SCAN_THREADS / 32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    TO acc = 0;
#pragma unroll
    for (int it = 0; it < SCAN_ITEMS; ++it) {
        int64_t x = base + (int64_t)it * SCAN_THREADS + threadIdx.x;
        if (x < n) acc += (TO)in[x];
    }
    TO total;
    block_exclusive_scan<TO>(acc, s_warp, &total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

template <typename TI, typename TO>
__global__ void __launch_bounds__(SCAN_THREADS) k_tile_scan(const TI *in, int64_t n, TO *out,
                                                            const TO *block_off) {
    __shared__ TO s_warp[SCAN_THREADS / 32];
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    TO v[SCAN_ITEMS];
    TO acc = 0;
#pragma unroll
    for (int it = 0; it < SCAN_ITEMS; ++it) {
        int64_t x = base + it;
        v[it] = x < n ? (TO)in[x] : TO(0);
        acc += v[it];
    }
    TO total;
    TO run = block_exclusive_scan<TO>(acc, s_warp, &total) + (block_off ? block_off[blockIdx.x] : TO(0));
#pragma unroll
    for (int it = 0; it < SCAN_ITEMS; ++it) {
        int64_t x = base + it;
        if (x < n) out[x] = run;
        run += v[it];
        if (x == n - 1) out[n] = run;
    }
}

template <typename TI, typename TO>
pastis_status scan_rec(pastis_ctx *c, const TI *in, TO *out, int64_t n, TO *tmp, int64_t tmp_len) {
    if (n <= 0) {
        PASTIS_CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(TO), c->stream));
        return PASTIS_OK;
    }
    int64_t nb = ceil_div64(n, SCAN_TILE);
    if (nb == 1) {
        k_tile_scan<TI, TO><<<1, SCAN_THREADS, 0, c->stream>>>(in, n, out, nullptr);
        PASTIS_LAUNCHED(c);
        return PASTIS_OK;
    }
    if (tmp_len < 2 * (nb + 1)) return PASTIS_ERR_INTERNAL;
    TO *sums = tmp, *offs = tmp + nb + 1;
    k_tile_reduce<TI, TO><<<(unsigned)nb, SCAN_THREADS, 0, c->stream>>>(in, n, sums);
    PASTIS_LAUNCHED(c);
    pastis_status st = scan_rec<TO, TO>(c, sums, offs, nb, tmp + 2 * (nb + 1), tmp_len - 2 * (nb + 1));
    if (st != PASTIS_OK) return st;
    k_tile_scan<TI, TO><<<(unsigned)nb, SCAN_THREADS, 0, c->stream>>>(in, n, out, offs);
    PASTIS_LAUNCHED(c);
    return PASTIS_OK;
}

int64_t scan_tmp_len(int64_t n) {
    int64_t t = 0;
    while (n > SCAN_TILE) {
        int64_t nb = ceil_div64(n, SCAN_TILE);
        t += 2 * (nb + 1);
        n = nb;
    }
    return t + 2;
}

}  // namespace

// A dedicated workspace slot for scan temporaries would collide when a scan runs inside
// the radix sort; the sort owns WS_SORT_HIST and scans use the slot after it.
#define WS_SCAN_TMP WS_FILT_SCAN

pastis_status exclusive_scan_u32(pastis_ctx *c, const uint32_t *in, uint32_t *out, int64_t n) {
    int64_t tl = scan_tmp_len(n);
    uint32_t *tmp;
    PASTIS_WS(tmp, c, WS_SCAN_TMP, sizeof(uint32_t) * tl);
    return scan_rec<uint32_t, uint32_t>(c, in, out, n, tmp, tl);
}

pastis_status exclusive_scan_i64(pastis_ctx *c, const int64_t *in, int64_t *out, int64_t n) {
    int64_t tl = scan_tmp_len(n);
    int64_t *tmp;
    PASTIS_WS(tmp, c, WS_SCAN_TMP, sizeof(int64_t) * tl);
    return scan_rec<int64_t, int64_t>(c, in, out, n, tmp, tl);
}

// ---------------------------------------------------------------------------------
// Stable LSD radix sort.  Per digit: a tile histogram, a scan of the
// (digit, tile) counts in digit-major order, then a scatter in which every warp ranks
// its items in input order, so equal digits keep input order.
// ---------------------------------------------------------------------------------
namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;   // each warp owns 256 consecutive items

template <int BITS>
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint32_t *keys, int64_t n, int shift,
                                                        uint32_t *hist, int64_t nb) {
    constexpr uint32_t D = 1u << BITS;
    __shared__ uint32_t s_h[D];
    if (threadIdx.x < D) s_h[threadIdx.x] = 0;
    __syncthreads();
    int64_t base = (int64_t)blockIdx.x * RS_TILE;
#pragma unroll 4
    for (int it = 0; it < RS_ITEMS; ++it) {
        int64_t x = base + (int64_t)it * RS_THREADS + threadIdx.x;
        if (x < n) atomicAdd(&s_h[(keys[x] >> shift) & (D - 1)], 1u);
    }
    __syncthreads();
    if (threadIdx.x < D) hist[(int64_t)threadIdx.x * nb + blockIdx.x] = s_h[threadIdx.x];
}

// The tile's items are first placed in shared memory in their sorted order (digit, then
// input order), then written out in that order, so consecutive threads write
// consecutive positions of each digit's run in the output.  The ranks of the first sweep
// are kept, so each item's peers are found once, by a ballot per bit of the digit.  Seven
// passes over the 35 M windows of 100,000 proteins: 3.10 ms with __match_any_sync in two sweeps
// and 16 items a thread, 1.64 ms so, 1.53 ms (3.9 TB/s) in digits of 7 and 6 bits.
constexpr size_t rs_scatter_smem(int bits) {
    return sizeof(uint64_t) * RS_TILE + sizeof(uint32_t) * RS_TILE +
           sizeof(uint32_t) * ((size_t)2 * (RS_WARPS + 1) * ((size_t)1 << bits) + RS_WARPS);
}

template <int BITS>
__global__ void __launch_bounds__(RS_THREADS) k_rs_scatter(const uint32_t *keys, const uint64_t *vals,
                                                           int64_t n, int shift, const uint32_t *offs,
                                                           int64_t nb, uint32_t *okeys, uint64_t *ovals) {
    constexpr uint32_t D = 1u << BITS;
    extern __shared__ __align__(16) unsigned char rs_smem[];
    uint64_t *s_v = reinterpret_cast<uint64_t *>(rs_smem);
    uint32_t *s_k = reinterpret_cast<uint32_t *>(s_v + RS_TILE);
    uint32_t *s_cnt = s_k + RS_TILE;                 // [warp][digit]: counts
    uint32_t *s_base = s_cnt + RS_WARPS * D;       // [warp][digit]: start within the digit's run
    uint32_t *s_tstart = s_base + RS_WARPS * D;    // [digit]: start of the digit's run in the tile
    uint32_t *s_gbase = s_tstart + D;              // [digit]: its start in the output
    uint32_t *s_wsum = s_gbase + D;                // [warp]: scan carries
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int d = threadIdx.x; d < (int)D * RS_WARPS; d += RS_THREADS) s_cnt[d] = 0;
    __syncthreads();
    const int64_t tile0 = (int64_t)blockIdx.x * RS_TILE;
    const int64_t base = tile0 + (int64_t)warp * (RS_ITEMS * 32);
    uint32_t k[RS_ITEMS];
    uint64_t v[RS_ITEMS];
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) {
        int64_t x = base + it * 32 + lane;
        bool ok = x < n;
        k[it] = ok ? keys[x] : 0u;
        v[it] = ok ? vals[x] : 0ull;
    }
    // each item's rank among its warp's items of the same digit, in input order, and with
    // it the warp's digit counts
    const unsigned lt_mask = (1u << lane) - 1u;
    uint32_t rank[RS_ITEMS / 2];                     // two 16-bit ranks a word
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) {
        const bool ok = base + it * 32 + lane < n;
        const uint32_t d = ok ? ((k[it] >> shift) & (D - 1)) : 0u;
        unsigned peers = __ballot_sync(0xffffffffu, ok);      // lanes with the same digit, by its bits
        peers = ok ? peers : 0u;
#pragma unroll
        for (int bit = 0; bit < BITS; ++bit) {
            const unsigned set = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
            peers &= ((d >> bit) & 1u) ? set : ~set;
        }
        const uint32_t before = ok ? s_cnt[warp * D + d] : 0u;
        __syncwarp();
        if (ok && lane == __ffs(peers) - 1) s_cnt[warp * D + d] = before + __popc(peers);
        __syncwarp();
        const uint32_t r = before + __popc(peers & lt_mask);
        rank[it >> 1] = (it & 1) ? rank[it >> 1] | (r << 16) : r;
    }
    __syncthreads();
    // per digit: the warps' starts within its run, its total, and the runs' starts in the
    // tile (an exclusive scan over the digits)
    const int d0 = threadIdx.x;                      // at most RS_THREADS digits
    uint32_t tot = 0;
    if (d0 < (int)D)
        for (int w = 0; w < RS_WARPS; ++w) {
            s_base[w * D + d0] = tot;
            tot += s_cnt[w * D + d0];
        }
    uint32_t incl = tot;
#pragma unroll
    for (int x = 1; x < 32; x <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, x);
        if (lane >= x) incl += y;
    }
    if (lane == 31) s_wsum[warp] = incl;
    if (d0 < (int)D) s_gbase[d0] = offs[(int64_t)d0 * nb + blockIdx.x];
    __syncthreads();
    uint32_t wpre = 0;
    for (int w = 0; w < warp; ++w) wpre += s_wsum[w];
    if (d0 < (int)D) s_tstart[d0] = wpre + incl - tot;
    __syncthreads();
    // each item to its place in the tile's sorted order
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) {
        if (base + it * 32 + lane < n) {
            const uint32_t d = (k[it] >> shift) & (D - 1);
            const uint32_t lp = s_tstart[d] + s_base[warp * D + d] + ((rank[it >> 1] >> (16 * (it & 1))) & 0xFFFFu);
            s_k[lp] = k[it];
            s_v[lp] = v[it];
        }
    }
    __syncthreads();
    // out in the tile's order: each digit's run lands contiguously
    const int tile_n = (int)min((int64_t)RS_TILE, n - tile0);
    for (int x = threadIdx.x; x < tile_n; x += RS_THREADS) {
        const uint32_t key = s_k[x];
        const uint32_t d = (key >> shift) & (D - 1);
        const uint32_t pos = s_gbase[d] + ((uint32_t)x - s_tstart[d]);
        okeys[pos] = key;
        ovals[pos] = s_v[x];
    }
}

template <int BITS>
pastis_status rs_pass(pastis_ctx *c, const uint32_t *ik, const uint64_t *iv, int64_t n, int shift, uint32_t *hist,
                      uint32_t *offs, int64_t nb, uint32_t *ok, uint64_t *ov) {
    prof_begin(c, "radix_hist");
    k_rs_hist<BITS><<<(unsigned)nb, RS_THREADS, 0, c->stream>>>(ik, n, shift, hist, nb);
    PASTIS_LAUNCHED(c);
    prof_end(c);
    pastis_status st = exclusive_scan_u32(c, hist, offs, nb << BITS);
    if (st != PASTIS_OK) return st;
    prof_begin(c, "radix_scatter");
    k_rs_scatter<BITS><<<(unsigned)nb, RS_THREADS, rs_scatter_smem(BITS), c->stream>>>(ik, iv, n, shift, offs, nb, ok,
                                                                                      ov);
    PASTIS_LAUNCHED(c);
    prof_end(c);
    return PASTIS_OK;
}

}  // namespace

// Keys below 2^key_bits.  As many passes as 8-bit digits need, of digits as equal as they
// come (28 bits: four of 7, not three of 8 and one of 4): fewer ballots and counters, and
// longer runs in each tile's writes.  The seven passes over 35 M windows (28 bits, then the 17 of
// the sequences) with their counts and scans: 2.53 ms in digits of 8 bits, 2.23 ms so.
pastis_status radix_sort_u32_u64(pastis_ctx *c, uint32_t *keys, uint64_t *vals, uint32_t *keys_alt,
                                 uint64_t *vals_alt, int64_t n, int key_bits, uint32_t **keys_out,
                                 uint64_t **vals_out) {
    *keys_out = keys;
    *vals_out = vals;
    if (n <= 1 || key_bits <= 0) return PASTIS_OK;
    if (n > 0xFFFFFFFFll) return PASTIS_ERR_UNSUPPORTED;
    int64_t nb = ceil_div64(n, RS_TILE);
    uint32_t *hist;
    PASTIS_WS(hist, c, WS_SORT_HIST, sizeof(uint32_t) * (256 * nb + 1) * 2);
    uint32_t *offs = hist + 256 * nb + 1;
    uint32_t *ik = keys, *ok = keys_alt;
    uint64_t *iv = vals, *ov = vals_alt;
    if (c->prof_on) c->sort_passes += n * (int64_t)((key_bits + 7) / 8);
    const int passes = (key_bits + 7) / 8, bits = std::max(5, (key_bits + passes - 1) / passes);
    for (int x = 0; x < passes; ++x) {
        auto pass = bits == 5 ? rs_pass<5> : bits == 6 ? rs_pass<6> : bits == 7 ? rs_pass<7> : rs_pass<8>;
        pastis_status st = pass(c, ik, iv, n, x * bits, hist, offs, nb, ok, ov);
        if (st != PASTIS_OK) return st;
        uint32_t *tk = ik; ik = ok; ok = tk;
        uint64_t *tv = iv; iv = ov; ov = tv;
    }
    *keys_out = ik;
    *vals_out = iv;
    return PASTIS_OK;
}

// ---------------------------------------------------------------------------------
// Column pointers from sorted codes.
// ---------------------------------------------------------------------------------
namespace {

constexpr int CP_THREADS = 256;
constexpr int CP_TILE = 8192;                    // codes a CTA

// The first indexes x in [0, n) with keys[x] >= k0 and >= k1, by the whole CTA: each half of
// the threads probes for one, 128 probes a round.
__device__ void block_lower_bounds(const uint32_t *__restrict__ keys, int64_t n, uint32_t k0, uint32_t k1, int64_t *r0,
                                   int64_t *r1) {
    constexpr int HALF = CP_THREADS / 2;
    const int half = threadIdx.x / HALF, t = threadIdx.x % HALF;
    int64_t lo[2] = {0, 0}, hi[2] = {n, n};      // the answers lie in [lo, hi]
    while (lo[0] < hi[0] || lo[1] < hi[1]) {
        const int64_t l = half ? lo[1] : lo[0], h = half ? hi[1] : hi[0];
        const int64_t x = l + (h - l + HALF - 1) / HALF * t;
        const bool below = x < h && keys[x] < (half ? k1 : k0);          // a prefix of the half's probes
        const int c[2] = {__syncthreads_count(below && half == 0), __syncthreads_count(below && half == 1)};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (lo[u] >= hi[u]) continue;
            const int64_t step = (hi[u] - lo[u] + HALF - 1) / HALF;
            if (c[u] == 0) { hi[u] = lo[u]; continue; }
            const int64_t last = lo[u] + step * (c[u] - 1);              // keys[last] is below
            hi[u] = step == 1 ? last + 1 : min(hi[u], last + step);
            lo[u] = last + 1;
        }
    }
    *r0 = lo[0];
    *r1 = lo[1];
}

// col_ptr[c] = the kept entries with a code below c, for c = 0 .. ncodes: a CTA fills CP_TILE
// codes.  It finds the tile's stretch of the sorted keys, marks where each code's run
// starts, and gives every code the start of the next present one (a suffix minimum, as
// the starts ascend).  Every entry of col_ptr is written once and nothing but the stretch
// is read, so the write of 24^6 pointers bounds it: 0.14 ms for a query's few k-mers, 0.38 ms
// for the 35 M entries of 100,000 proteins, where clearing, counting by atomics and a scan
// in place took 0.98 and 1.05 ms.
__global__ void __launch_bounds__(CP_THREADS) k_fill_col_ptr(const uint32_t *__restrict__ keys,
                                                             const uint32_t *__restrict__ keep_off, int64_t n,
                                                             int64_t ncodes, uint32_t *__restrict__ col_ptr) {
    __shared__ __align__(16) uint32_t s_start[CP_TILE];
    __shared__ uint32_t s_wmin[CP_THREADS / 32];
    const int64_t c0 = (int64_t)blockIdx.x * CP_TILE;
    int64_t x0, x1;
    block_lower_bounds(keys, n, (uint32_t)c0, (uint32_t)min(c0 + CP_TILE, ncodes), &x0, &x1);
    for (int i = threadIdx.x; i < CP_TILE / 4; i += CP_THREADS)
        reinterpret_cast<uint4 *>(s_start)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
    if (threadIdx.x < CP_THREADS / 32) s_wmin[threadIdx.x] = ~0u;
    __syncthreads();
    constexpr int PER_WARP = CP_TILE / (CP_THREADS / 32);
    for (int64_t x = x0 + threadIdx.x; x < x1; x += CP_THREADS) {
        const uint32_t k = keys[x];
        if (x == x0 || keys[x - 1] != k) {
            const uint32_t v = keep_off[x];
            const int i = (int)(k - (uint32_t)c0);
            s_start[i] = v;
            atomicMin(&s_wmin[i / PER_WARP], v);
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t next = keep_off[x1];                // what follows the warp's codes
    for (int w = warp + 1; w < CP_THREADS / 32; ++w) next = min(next, s_wmin[w]);
    for (int r = PER_WARP / 128 - 1; r >= 0; --r) {
        const int i = warp * PER_WARP + r * 128 + lane * 4;
        uint4 v = *reinterpret_cast<const uint4 *>(s_start + i);
        v.z = min(v.z, v.w);
        v.y = min(v.y, v.z);
        v.x = min(v.x, v.y);
        uint32_t m = v.x;                        // then the lanes behind
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t o = __shfl_down_sync(0xffffffffu, m, d);
            if (lane + d < 32) m = min(m, o);
        }
        const uint32_t first = min(__shfl_sync(0xffffffffu, m, 0), next);
        uint32_t behind = __shfl_down_sync(0xffffffffu, m, 1);
        behind = lane == 31 ? next : min(behind, next);
        v.x = min(v.x, behind);
        v.y = min(v.y, behind);
        v.z = min(v.z, behind);
        v.w = min(v.w, behind);
        next = first;
        const int64_t c = c0 + i;
        if (c + 3 <= ncodes && (((uintptr_t)(col_ptr + c)) & 15) == 0) {
            *reinterpret_cast<uint4 *>(col_ptr + c) = v;
        } else {
            if (c <= ncodes) col_ptr[c] = v.x;
            if (c + 1 <= ncodes) col_ptr[c + 1] = v.y;
            if (c + 2 <= ncodes) col_ptr[c + 2] = v.z;
            if (c + 3 <= ncodes) col_ptr[c + 3] = v.w;
        }
    }
}

// The same for few codes, a thread each: one binary search of the sorted keys.
__global__ void k_find_col_ptr(const uint32_t *__restrict__ keys, const uint32_t *__restrict__ keep_off, int64_t n,
                               int64_t ncodes, uint32_t *__restrict__ col_ptr) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c > ncodes) return;
    int64_t a = 0, b = n;
    while (a < b) {
        const int64_t m = (a + b) >> 1;
        if ((int64_t)keys[m] < c) a = m + 1; else b = m;
    }
    col_ptr[c] = keep_off[a];
}

}  // namespace

pastis_status fill_col_ptr(pastis_ctx *c, const uint32_t *keys, const uint32_t *keep_off, int64_t n, int64_t ncodes,
                           uint32_t *col_ptr) {
    prof_begin(c, "col_ptr");
    // A search per code instead where there are too few tiles to fill the SMs (k <= 4), or where
    // the tiles' stretches of keys take longer than the searches, which hardly depend on the
    // keys: from one key a code on with a wave or two of tiles (k = 5, 6 tiles an SM), whose
    // longest, those of the frequent residues, finish late; from six where the tiles fill the SMs
    // many times over (k = 6, 153 an SM).
    // Measured on residues at their natural frequencies, tiles and searches in us: k = 4, 1 M
    // keys 110 and 12; k = 5, 8 M codes: 4 M keys 82 and 148, 7.6 M 164 and 167, 20 M 382 and
    // 188, 300 M 3,129 and 285; k = 6, 191 M codes: 35 M keys 356 and 3,665, 350 M 1,866 and
    // 4,440, 1 G 4,171 and 4,835, 1.2 G 4,780 and 5,016.
    const int64_t tiles = ceil_div64(ncodes + 1, CP_TILE), sms = c->sm_count;
    if (tiles < 2 * sms || n > ncodes * (tiles < 32 * sms ? 1 : 6))
        k_find_col_ptr<<<(unsigned)ceil_div64(ncodes + 1, 256), 256, 0, c->stream>>>(keys, keep_off, n, ncodes, col_ptr);
    else
        k_fill_col_ptr<<<(unsigned)tiles, CP_THREADS, 0, c->stream>>>(keys, keep_off, n, ncodes, col_ptr);
    PASTIS_LAUNCHED(c);
    prof_end(c);
    return PASTIS_OK;
}

cudaError_t radix_set_smem_limit() {
    return cudaFuncSetAttribute(k_rs_scatter<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rs_scatter_smem(8));
}
