// Learned prefilter: a 16 -> 256 -> 256 -> 1 MLP over per-pair features that predicts
// whether a candidate pair's alignment will pass the similarity filter (Sec. IV-F), so
// that pairs predicted to fail skip the alignment.  The exact path stays the reference:
// labels come from it, and the kept fraction and edge recall are measured against it.
// (The paper's own lever for fewer alignments is the common-k-mer threshold, Sec. VI,
// which costs 2-3% recall; this is a learned version of the same trade.)
//
// Features (16, float32 -> bf16): log1p(count), the two seed diagonals (pos_i - pos_j)
// scaled by 1/256, their spread, log lengths of i and j, log min/max length, the length
// ratio, the BLOSUM scores of the two seed k-mers and their sum (/ 32), count / shorter
// length, seed-1-present flag, and zeros to 16.
//
// Arithmetic: bf16 weights and activations, float32 accumulation on the tensor cores
// (mma.sync m16n8k16, bf16 inputs, f32 accumulators), float32 master weights and Adam
// moments.  One kernel runs the network forward (in training also back to layer 1), one
// forms the gradients of W1 and W2, one sums the others and takes the Adam step.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "internal.cuh"

namespace {

constexpr int FEAT = 16, HID = 256;

__device__ __forceinline__ float bf(const __nv_bfloat16 v) { return __bfloat162float(v); }

// ---------------------------------------------------------------------------------
// features
// ---------------------------------------------------------------------------------
__global__ void k_pair_features(const uint8_t *qcodes, const int64_t *qoffsets, const uint8_t *tcodes,
                                const int64_t *toffsets, const pastis_cand *pairs, int64_t n, int k,
                                const int8_t *gmat, __nv_bfloat16 *x) {
    int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    const pastis_cand c = pairs[p];
    const int64_t qo = qoffsets[c.i], to = toffsets[c.j];
    const float lq = (float)(qoffsets[c.i + 1] - qo), lt = (float)(toffsets[c.j + 1] - to);
    float f[FEAT];
#pragma unroll
    for (int t = 0; t < FEAT; ++t) f[t] = 0.f;
    const bool two = c.qpos[1] != 0xFFFF;
    const float d0 = (float)c.qpos[0] - (float)c.tpos[0];
    const float d1 = two ? (float)c.qpos[1] - (float)c.tpos[1] : d0;
    float s0 = 0.f, s1 = 0.f;
    for (int t = 0; t < k; ++t) {
        s0 += gmat[qcodes[qo + c.qpos[0] + t] * PASTIS_NSYM + tcodes[to + c.tpos[0] + t]];
        if (two) s1 += gmat[qcodes[qo + c.qpos[1] + t] * PASTIS_NSYM + tcodes[to + c.tpos[1] + t]];
    }
    const float mn = fminf(lq, lt), mx = fmaxf(lq, lt);
    f[0] = log1pf((float)c.count);
    f[1] = d0 / 256.f;
    f[2] = d1 / 256.f;
    f[3] = fabsf(d0 - d1) / 256.f;
    f[4] = logf(lq + 1.f);
    f[5] = logf(lt + 1.f);
    f[6] = logf(mn + 1.f);
    f[7] = logf(mx + 1.f);
    f[8] = mn / fmaxf(mx, 1.f);
    f[9] = s0 / 32.f;
    f[10] = s1 / 32.f;
    f[11] = (s0 + s1) / 32.f;
    f[12] = (float)c.count / fmaxf(mn, 1.f);
    f[13] = two ? 1.f : 0.f;
#pragma unroll
    for (int t = 0; t < FEAT; ++t) x[p * FEAT + t] = __float2bfloat16(f[t]);
}

// ---------------------------------------------------------------------------------
// The network: one persistent kernel takes 64 rows at a time through all three layers
// (and, in training, back to the gradient at layer 1), with the activations in shared
// memory.  A CTA's two groups of eight warps each work on a tile of their own, so one's
// epilogues run under the other's products.  W2 stays there for the kernel's life, in rows of 256 + 8 values so that the
// eight rows of an ldmatrix lie in different banks.  A warp owns 32 rows x 64 columns of
// every product; the k steps of 16 run in order from a zero accumulator, so a logit does
// not depend on the batch it is computed in.
// What bounds it is the rate of mma.sync with every operand fragment read from shared
// memory.  mma.sync, not tcgen05: its sums are the ones the selection thresholds in use
// were calibrated on, and a step of the path spends about 1% here.
// ---------------------------------------------------------------------------------
constexpr int TM = 64;                               // rows of a tile
constexpr int MLP_GROUPS = 2;                        // groups of eight warps, a tile each
constexpr int LDH = HID + 8, LDX = FEAT + 8;         // row pitches in shared memory
constexpr int GROUP = 256, MLP_THREADS = MLP_GROUPS * GROUP;
constexpr int PART = 3 * HID;                        // a slot's partial sums: g_b1, g_b2, g_w3
constexpr int MLP_SLOTS = 152;                       // slots at most, a CTA each where there are as many SMs
constexpr size_t MLP_SMEM = sizeof(__nv_bfloat16) * ((size_t)HID * LDH + FEAT * LDH + MLP_GROUPS * (TM * LDH + TM * LDX)) +
                            sizeof(float) * 3 * HID;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two columns of a fragment as they are stored: relu(acc + bias) in bf16.
__device__ __forceinline__ uint32_t bias_relu2(float v0, float v1, const float *bias) {
    __nv_bfloat162 h;
    h.x = __float2bfloat16(fmaxf(v0 + bias[0], 0.f));
    h.y = __float2bfloat16(fmaxf(v1 + bias[1], 0.f));
    return *reinterpret_cast<uint32_t *>(&h);
}
// Eight bf16 from memory that may not be 16-byte aligned (the caller's buffers).
__device__ __forceinline__ uint4 load8(const __nv_bfloat16 *p, bool aligned) {
    if (aligned) return *reinterpret_cast<const uint4 *>(p);
    const uint16_t *q = reinterpret_cast<const uint16_t *>(p);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = (uint32_t)q[2 * i] | ((uint32_t)q[2 * i + 1] << 16);
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// acc[2][8][4] = the warp's 32 rows (mw) x 64 columns (nw) of s_h (bf16, 64 x 256) times
// W2 (TW: its transpose).
template <bool TW>
__device__ __forceinline__ void tile_product(float (&acc)[2][8][4], uint32_t h, uint32_t w2, int mw, int nw, int lane) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][t][q] = 0.f;
    const uint32_t ha = h + (uint32_t)(((mw * 32 + (lane & 15)) * LDH + (lane >> 4) * 8) * 2);
    const uint32_t wb = TW ? w2 + (uint32_t)(((nw * 64 + (lane & 7) + ((lane >> 4) << 3)) * LDH + ((lane >> 3) & 1) * 8) * 2)
                           : w2 + (uint32_t)(((lane & 15) * LDH + nw * 64 + (lane >> 4) * 8) * 2);
#pragma unroll 2
    for (int k = 0; k < HID; k += 16) {
        uint32_t a[2][4];
        ldsm4(a[0], ha + k * 2);
        ldsm4(a[1], ha + (16 * LDH + k) * 2);
#pragma unroll
        for (int t = 0; t < 8; t += 2) {
            uint32_t b[4];
            if (TW) ldsm4(b, wb + (t * 8 * LDH + k) * 2);
            else ldsm4t(b, wb + (k * LDH + t * 8) * 2);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                mma16816(acc[i][t], a[i], b[0], b[1]);
                mma16816(acc[i][t + 1], a[i], b[2], b[3]);
            }
        }
    }
}

struct mlp_w {
    const __nv_bfloat16 *w1, *w2, *w3;
    const float *b1, *b2, *b3;
};
struct mlp_train_io {           // training only
    const float *y;
    float pos_weight;
    __nv_bfloat16 *h1, *dh1, *dh2;   // n x 256 each, for the gradients of W1 and W2
    float *dz, *lrow;           // per row: the gradient at the logit, the loss term
    float *part;                // PART floats per slot
    int slots;
};

// z[r] = the logit of row r.  TRAIN: the weighted logistic loss's terms and dz = w *
// (sigmoid(z) - y) / n instead, the gradients dh2 = dz * w3 where layer 2 is active and dh1 = dh2 W2^T where
// layer 1 is, and the gradients of W3 and its layers' biases as partial sums per slot: the tiles go
// to min(tiles, MLP_SLOTS) slots in turn, whatever the number of CTAs, and k_mlp_adam adds the
// slots in order, so a training step gives the same bits on any number of SMs.  Measured on 10^6 rows: 3.99 ms with
// one 64 x 64 tile and 2-byte loads a CTA and h1, h2 through memory, 0.355 ms so (137 GF:
// 0.6 of the rate mma.sync reaches alone); a training step of 65,536 rows 28.1 ms with the
// column sums in one CTA each, 0.35 ms so.
template <bool TRAIN>
__global__ void __launch_bounds__(MLP_THREADS, 1) k_mlp(mlp_w net, const __nv_bfloat16 *__restrict__ x, int64_t n,
                                                        float *__restrict__ z, mlp_train_io tr) {
    const int lane = threadIdx.x & 31, group = threadIdx.x / GROUP;
    const int tid = threadIdx.x % GROUP, warp = tid >> 5;                // within the group
    const int gid = lane >> 2, tig = lane & 3;
    const int mw = warp >> 2, nw = warp & 3;             // the warp's 32 rows x 64 columns
    auto sync = [group]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(GROUP) : "memory"); };
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    __nv_bfloat16 *s_w2 = reinterpret_cast<__nv_bfloat16 *>(mlp_smem);   // [256][LDH], input-major
    __nv_bfloat16 *s_w1 = s_w2 + HID * LDH;                              // [16][LDH]
    __nv_bfloat16 *s_h = s_w1 + FEAT * LDH + group * TM * LDH;           // [64][LDH]: h1, then h2, dh2, dh1
    __nv_bfloat16 *s_x = s_w1 + FEAT * LDH + MLP_GROUPS * TM * LDH + group * TM * LDX;   // [64][LDX]
    float *s_b1 = reinterpret_cast<float *>(s_w1 + FEAT * LDH + MLP_GROUPS * TM * (LDH + LDX));
    float *s_b2 = s_b1 + HID, *s_w3 = s_b2 + HID;
    const bool wal = ((((uintptr_t)net.w1) | ((uintptr_t)net.w2)) & 15) == 0, xal = (((uintptr_t)x) & 15) == 0;
    for (int i = threadIdx.x; i < (HID + FEAT) * HID / 8; i += MLP_THREADS) {
        const int r = i >> 5, c = (i & 31) * 8;
        const uint4 v = r < HID ? load8(net.w2 + r * HID + c, wal) : load8(net.w1 + (r - HID) * HID + c, wal);
        *reinterpret_cast<uint4 *>(s_w2 + r * LDH + c) = v;              // W1's rows follow W2's
    }
    if (group == 0) {
        s_b1[tid] = net.b1[tid];
        s_b2[tid] = net.b2[tid];
        s_w3[tid] = bf(net.w3[tid]);
    }
    __syncthreads();
    const float b3 = net.b3[0];
    const uint32_t u_h = smem_u32(s_h), u_w1 = smem_u32(s_w1), u_w2 = smem_u32(s_w2), u_x = smem_u32(s_x);
    const int64_t tiles = (n + TM - 1) / TM;
    const int xr = tid >> 1, xc = (tid & 1) * 8;         // 128 threads load 8 features of a tile each
    auto load_x = [&](int64_t tile) {
        const int64_t r = tile * TM + xr;
        return xr < TM && tile < tiles && r < n ? load8(x + r * FEAT + xc, xal) : make_uint4(0u, 0u, 0u, 0u);
    };
    const int slots = TRAIN ? tr.slots : (int)gridDim.x;
    for (int slot = blockIdx.x; slot < slots; slot += gridDim.x) {
        // TRAIN: sums kept over the slot's tiles
        float gw3[8], gb2[8], gb1[16];
        if constexpr (TRAIN) {
#pragma unroll
            for (int t = 0; t < 8; ++t) { gw3[t] = 0.f; gb2[t] = 0.f; }
#pragma unroll
            for (int t = 0; t < 16; ++t) gb1[t] = 0.f;
        }
        const int64_t step = (int64_t)slots * MLP_GROUPS, tile0 = (int64_t)group * slots + slot;
        uint4 xv = load_x(tile0);
        for (int64_t tile = tile0; tile < tiles; tile += step) {
            const int64_t r0 = tile * TM;
            if (xr < TM) *reinterpret_cast<uint4 *>(s_x + xr * LDX + xc) = xv;
            sync();                                          // x here; the group is done with its last tile
            xv = load_x(tile + step);
            // layer 1: one k step
            uint32_t act[2] = {0u, 0u};                      // TRAIN: which of the warp's fragment values are active
            {
                uint32_t a[2][4];
                ldsm4(a[0], u_x + (uint32_t)(((mw * 32 + (lane & 15)) * LDX + (lane >> 4) * 8) * 2));
                ldsm4(a[1], u_x + (uint32_t)(((mw * 32 + 16 + (lane & 15)) * LDX + (lane >> 4) * 8) * 2));
#pragma unroll
                for (int t = 0; t < 8; t += 2) {
                    uint32_t b[4];
                    ldsm4t(b, u_w1 + (uint32_t)(((lane & 15) * LDH + nw * 64 + t * 8 + (lane >> 4) * 8) * 2));
#pragma unroll
                    for (int i = 0; i < 2; ++i)
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            float c[4] = {0.f, 0.f, 0.f, 0.f};
                            mma16816(c, a[i], b[2 * u], b[2 * u + 1]);
                            const int col = nw * 64 + (t + u) * 8 + tig * 2, row = mw * 32 + i * 16 + gid;
                            const uint32_t lo = bias_relu2(c[0], c[1], s_b1 + col), hi = bias_relu2(c[2], c[3], s_b1 + col);
                            *reinterpret_cast<uint32_t *>(s_h + row * LDH + col) = lo;
                            *reinterpret_cast<uint32_t *>(s_h + (row + 8) * LDH + col) = hi;
                            if constexpr (TRAIN) {           // stored halves are never negative: non-zero is active
                                const uint32_t m = ((lo & 0x7FFFu) ? 1u : 0u) | ((lo & 0x7FFF0000u) ? 2u : 0u) |
                                                   ((hi & 0x7FFFu) ? 4u : 0u) | ((hi & 0x7FFF0000u) ? 8u : 0u);
                                act[i] |= m << (4 * (t + u));
                            }
                        }
                }
            }
            sync();
            if constexpr (TRAIN)
                for (int i = tid; i < TM * (HID / 8); i += GROUP) {
                    const int64_t r = r0 + (i >> 5);
                    if (r < n)
                        *reinterpret_cast<uint4 *>(tr.h1 + r * HID + (i & 31) * 8) =
                            *reinterpret_cast<const uint4 *>(s_h + (i >> 5) * LDH + (i & 31) * 8);
                }
            float acc[2][8][4];
            tile_product<false>(acc, u_h, u_w2, mw, nw, lane);
            sync();                                 // h1 is read: h2 takes its place
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    const int col = nw * 64 + t * 8 + tig * 2, row = mw * 32 + i * 16 + gid;
                    *reinterpret_cast<uint32_t *>(s_h + row * LDH + col) = bias_relu2(acc[i][t][0], acc[i][t][1], s_b2 + col);
                    *reinterpret_cast<uint32_t *>(s_h + (row + 8) * LDH + col) =
                        bias_relu2(acc[i][t][2], acc[i][t][3], s_b2 + col);
                }
            sync();
            // the head: a warp takes 16 rows, a lane every 32nd column
#pragma unroll 2
            for (int q = 0; q < TM / 8; ++q) {
                const int row = warp * (TM / 8) + q;
                float h[8], s = 0.f;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    h[t] = bf(s_h[row * LDH + lane + 32 * t]);
                    s += h[t] * s_w3[lane + 32 * t];
                }
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
                const float zz = s + b3;
                if (!TRAIN && r0 + row < n && lane == 0) z[r0 + row] = zz;
                if constexpr (TRAIN) {
                    float d = 0.f;
                    if (r0 + row < n) {
                        const float yy = tr.y[r0 + row];
                        const float w = yy > 0.5f ? tr.pos_weight : 1.f;
                        const float sg = 1.f / (1.f + __expf(-zz));
                        d = w * (sg - yy) / (float)n;
                        const float sp = zz > 0.f ? zz + log1pf(__expf(-zz)) : log1pf(__expf(zz));
                        if (lane == 0) {
                            tr.dz[r0 + row] = d;
                            tr.lrow[r0 + row] = w * (sp - yy * zz) / (float)n;
                        }
                    }
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        const bool on = r0 + row < n && h[t] > 0.f;
                        const __nv_bfloat16 dv = __float2bfloat16(on ? d * s_w3[lane + 32 * t] : 0.f);
                        s_h[row * LDH + lane + 32 * t] = dv;
                        gw3[t] += h[t] * d;              // d = 0 past the batch
                        gb2[t] += bf(dv);
                    }
                }
            }
            if constexpr (TRAIN) {
                sync();
                for (int i = tid; i < TM * (HID / 8); i += GROUP) {
                    const int64_t r = r0 + (i >> 5);
                    if (r < n)
                        *reinterpret_cast<uint4 *>(tr.dh2 + r * HID + (i & 31) * 8) =
                            *reinterpret_cast<const uint4 *>(s_h + (i >> 5) * LDH + (i & 31) * 8);
                }
                tile_product<true>(acc, u_h, u_w2, mw, nw, lane);
                sync();                             // dh2 is read: dh1 takes its place
#pragma unroll
                for (int t = 0; t < 8; ++t) {
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        const int col = nw * 64 + t * 8 + tig * 2, row = mw * 32 + i * 16 + gid;
                        const uint32_t m = act[i] >> (4 * t);
                        float v[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) v[q] = (m >> q) & 1u ? acc[i][t][q] : 0.f;
                        gb1[2 * t] += v[0] + v[2];
                        gb1[2 * t + 1] += v[1] + v[3];
                        __nv_bfloat162 p0, p1;
                        p0.x = __float2bfloat16(v[0]); p0.y = __float2bfloat16(v[1]);
                        p1.x = __float2bfloat16(v[2]); p1.y = __float2bfloat16(v[3]);
                        *reinterpret_cast<__nv_bfloat162 *>(s_h + row * LDH + col) = p0;
                        *reinterpret_cast<__nv_bfloat162 *>(s_h + (row + 8) * LDH + col) = p1;
                    }
                }
                sync();
                for (int i = tid; i < TM * (HID / 8); i += GROUP) {
                    const int64_t r = r0 + (i >> 5);
                    if (r < n)
                        *reinterpret_cast<uint4 *>(tr.dh1 + r * HID + (i & 31) * 8) =
                            *reinterpret_cast<const uint4 *>(s_h + (i >> 5) * LDH + (i & 31) * 8);
                }
            }
            sync();                                 // s_x and s_h are free
        }
        if constexpr (TRAIN) {
            // the slot's partial sums, through shared memory: [16 warps][256] g_b2, the same g_w3,
            // [2 groups x 2][256] g_b1
            __syncthreads();
            constexpr int W = MLP_THREADS / 32;
            const int aw = threadIdx.x >> 5;
            float *part = tr.part + (int64_t)slot * PART;
            float *s_red = reinterpret_cast<float *>(s_w1 + FEAT * LDH);
#pragma unroll
            for (int t = 0; t < 8; ++t) {
                s_red[aw * HID + lane + 32 * t] = gb2[t];
                s_red[(W + aw) * HID + lane + 32 * t] = gw3[t];
            }
#pragma unroll
            for (int t = 0; t < 16; ++t) {                   // over the eight rows' lanes of a column
                float v = gb1[t];
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (gid == 0) s_red[(2 * W + group * 2 + mw) * HID + nw * 64 + (t >> 1) * 8 + tig * 2 + (t & 1)] = v;
            }
            __syncthreads();
            if (group == 0) {
                float a = 0.f, b = 0.f, c = 0.f;
                for (int w = 0; w < W; ++w) { a += s_red[w * HID + tid]; b += s_red[(W + w) * HID + tid]; }
                for (int w = 0; w < 2 * MLP_GROUPS; ++w) c += s_red[(2 * W + w) * HID + tid];
                part[tid] = c;
                part[HID + tid] = a;
                part[2 * HID + tid] = b;
            }
            __syncthreads();                        // the next slot's tiles take their place
        }
        if constexpr (!TRAIN) break;                // a slot a CTA
    }
}

// The gradients of W2 (h1^T dh2) and W1 (x^T dh1): every entry is one chain of mma.sync over
// the rows, 16 at a time in order, so what bounds it is the time of a step through the
// 4,096 of a 65,536-row batch: the fragments of a stage are read from the ring of cp.async stages
// while the products of the one before run.  The chains run side by side, 32 inputs x 32
// outputs a CTA (two chains a warp), 64 CTAs for W2 and 8 for W1, each reading only its
// columns.  Tiles of 64 x 64 with 2-byte loads took 16.8 ms of a 65,536-row step, 0.23 ms with
// read and product one after the other, 0.197 ms so (stages of 128 rows 0.210, rings of 5, 14
// and 20 stages 0.266, 0.208 and 0.208); chains split over the rows and added up would be
// faster still, but the sums would differ from these by more than a re-ordering (3e-4: the
// tensor core truncates what it aligns to a long chain's accumulator).
constexpr int WG_ROWS = 64, WG_STAGES = 8, WG_COLS = 32, LDG = WG_COLS + 8;
constexpr int WG_PROD = 128, WG_THREADS = WG_PROD + 256;   // four warps of products, then eight that fetch
constexpr int WG_STAGE = 2 * WG_ROWS * LDG;              // bf16 values of a stage
constexpr size_t WG_SMEM = sizeof(__nv_bfloat16) * WG_STAGES * WG_STAGE;

constexpr int WG_CTAS = 64 + 8 + 1;

// The sums of dz (W3's bias) and of the loss terms over the rows, by the last CTA beside the
// chains: every 256th row to a thread, then a tree, so their rounding does not depend on
// the number of SMs.
__device__ void row_sums(const float *__restrict__ dz, const float *__restrict__ lrow, int64_t n, float *g_b3,
                         float *loss, float *s) {
    const int t = threadIdx.x;
    if (t < 256) {
        float a = 0.f, b = 0.f;
#pragma unroll 8
        for (int64_t r = t; r < n; r += 256) { a += dz[r]; b += lrow[r]; }
        s[t] = a;
        s[256 + t] = b;
    }
    __syncthreads();
    for (int d = 128; d > 0; d >>= 1) {
        if (t < d) { s[t] += s[t + d]; s[256 + t] += s[256 + t + d]; }
        __syncthreads();
    }
    if (t == 0) {
        *g_b3 = s[0];
        if (loss) *loss = s[256];
    }
}

__global__ void __launch_bounds__(WG_THREADS, 1) k_mlp_wgrad(const __nv_bfloat16 *__restrict__ x,
                                                          const __nv_bfloat16 *__restrict__ h1,
                                                          const __nv_bfloat16 *__restrict__ dh1,
                                                          const __nv_bfloat16 *__restrict__ dh2, int64_t n,
                                                          const float *__restrict__ dz,
                                                          const float *__restrict__ lrow, float *__restrict__ g_w1,
                                                          float *__restrict__ g_w2, float *__restrict__ g_b3,
                                                          float *__restrict__ loss) {
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    __nv_bfloat16 *s = reinterpret_cast<__nv_bfloat16 *>(mlp_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mw = (warp >> 1) & 1, nw = warp & 1;       // a product warp's 16 x 16 entries
    if (blockIdx.x == WG_CTAS - 1) {
        row_sums(dz, lrow, n, g_b3, loss, reinterpret_cast<float *>(mlp_smem));
        return;
    }
    const bool first = blockIdx.x >= 64;                 // W1
    const int i0 = first ? 0 : (blockIdx.x >> 3) * WG_COLS, o0 = (blockIdx.x & 7) * WG_COLS;
    const int stages = (int)((n + WG_ROWS - 1) / WG_ROWS);
    float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    if (warp >= WG_PROD / 32) {
        // warps 4 .. 11 fetch: a thread always takes the same 16-byte piece of a row, of A or of
        // B, from every 32nd row; W1's A has two pieces, W2's four
        const __nv_bfloat16 *A = first ? x : h1 + i0, *B = (first ? dh1 : dh2) + o0;
        const int t = threadIdx.x - WG_PROD, c = t & 7, row0 = t >> 3;
        const bool from_b = c >= 4, mine = from_b || c < (first ? FEAT / 8 : WG_COLS / 8);
        const int ld = !from_b && first ? FEAT : HID;
        const __nv_bfloat16 *src = (from_b ? B + (c - 4) * 8 : A + (mine ? c * 8 : 0)) + (int64_t)row0 * ld;
        const bool aligned = (((uintptr_t)src) & 15) == 0;               // x is the caller's
        __nv_bfloat16 *const dst = s + (from_b ? WG_ROWS * LDG + (c - 4) * 8 : c * 8) + row0 * LDG;
        int left = (int)n - row0;                        // rows from this thread's next one on
        int put = 0;                                     // ring slot of the next fetch
        auto fetch = [&]() {
            if (mine) {
                __nv_bfloat16 *d = dst + put * WG_STAGE;
                const uint32_t d32 = smem_u32(d);
                if (aligned && left > WG_ROWS - 32) {
#pragma unroll
                    for (int u = 0; u < WG_ROWS / 32; ++u)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d32 + u * 32 * LDG * 2),
                                     "l"(src + u * 32 * ld));
                } else {                                 // rows past the batch are zero
#pragma unroll
                    for (int u = 0; u < WG_ROWS / 32; ++u)
                        *reinterpret_cast<uint4 *>(d + u * 32 * LDG) =
                            left > u * 32 ? load8(src + u * 32 * ld, aligned) : make_uint4(0u, 0u, 0u, 0u);
                }
            }
            src += (int64_t)WG_ROWS * ld;
            left -= WG_ROWS;
            put = put + 1 == WG_STAGES ? 0 : put + 1;
            asm volatile("cp.async.commit_group;");
        };
#pragma unroll
        for (int st = 0; st < WG_STAGES - 2; ++st) fetch();
        for (int st = 0; st < stages; ++st) {
            asm volatile("cp.async.wait_group %0;" ::"n"(WG_STAGES - 3));
            __syncthreads();                             // stage st is here, and stage st - 2 is used
            fetch();
        }
        asm volatile("cp.async.wait_group 0;");
        return;
    }
    const int q = lane >> 3;
    const uint32_t a_at = smem_u32(s) + (uint32_t)((((lane & 7) + (q >> 1) * 8) * LDG + mw * 16 + (q & 1) * 8) * 2);
    const uint32_t b_at = smem_u32(s) + (uint32_t)((WG_ROWS * LDG + (lane & 15) * LDG + nw * 16 + (lane >> 4) * 8) * 2);
    uint32_t at = 0;                                     // byte offset of the stage in the ring
    int rows = (int)n;                                   // rows from the stage to multiply on
    const bool works = !(first && mw == 1);              // W1 has 16 inputs
    // the fragments of a stage are read while the products of the one before run
    uint32_t fa[2][WG_ROWS / 16][4], fb[2][WG_ROWS / 16][4];
    auto read = [&](uint32_t (&a)[WG_ROWS / 16][4], uint32_t (&b)[WG_ROWS / 16][4]) {
        __syncthreads();
        if (works)
#pragma unroll
            for (int k = 0; k < WG_ROWS / 16; ++k) {
                ldsm4t(a[k], a_at + at + k * 16 * LDG * 2);
                ldsm4t(b[k], b_at + at + k * 16 * LDG * 2);
            }
        at = at + WG_STAGE * 2 == WG_STAGES * WG_STAGE * 2 ? 0u : at + WG_STAGE * 2;
    };
    auto multiply = [&](uint32_t (&a)[WG_ROWS / 16][4], uint32_t (&b)[WG_ROWS / 16][4]) {
        if (works)
#pragma unroll
            for (int k = 0; k < WG_ROWS / 16; ++k)
                if (k * 16 < rows) {
                    mma16816(acc[0], a[k], b[k][0], b[k][1]);
                    mma16816(acc[1], a[k], b[k][2], b[k][3]);
                }
        rows -= WG_ROWS;
    };
    read(fa[0], fb[0]);
    int st = 1;
    for (; st + 1 < stages; st += 2) {
        read(fa[1], fb[1]);
        multiply(fa[0], fb[0]);
        read(fa[0], fb[0]);
        multiply(fa[1], fb[1]);
    }
    if (st < stages) {
        read(fa[1], fb[1]);
        multiply(fa[0], fb[0]);
        multiply(fa[1], fb[1]);
    } else {
        multiply(fa[0], fb[0]);
    }
    if (first && mw == 1) return;
    float *out = first ? g_w1 : g_w2;
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q)
            out[(i0 + mw * 16 + (lane >> 2) + (q >> 1) * 8) * HID + o0 + nw * 16 + t * 8 + (lane & 3) * 2 + (q & 1)] =
                acc[t][q];
}

// Every parameter's Adam step on its float32 master, with the gradients of W3 and of the
// biases of layers 1 and 2 summed here from the slots' partial sums (in order); refreshes the
// bf16 copies.
struct adam_args {
    float *w1, *b1, *w2, *b2, *w3, *b3;
    __nv_bfloat16 *w1b, *w2b, *w3b;
    float *grad, *m, *v;
    float lr, beta1, beta2, eps, c1, c2;
};

__global__ void __launch_bounds__(256) k_mlp_adam(adam_args a, const float *__restrict__ part, int n_part) {
    constexpr int NW1 = FEAT * HID, NW2 = HID * HID, O1 = NW1, O2 = O1 + HID, O3 = O2 + NW2, O4 = O3 + HID,
                  O5 = O4 + HID, N = O5 + 1;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= N) return;
    float g;
    if (x < O1 || (x >= O2 && x < O3) || x == O5) {
        g = a.grad[x];
    } else {
        const float *p = part + (x < O2 ? x - O1 : x - O3 + HID);     // b1, then b2, w3
        g = 0.f;
#pragma unroll 8
        for (int q = 0; q < n_part; ++q) g += p[q * PART];
        a.grad[x] = g;
    }
    float *w;
    __nv_bfloat16 *wb = nullptr;
    if (x < O1) { w = a.w1 + x; wb = a.w1b + x; }
    else if (x < O2) w = a.b1 + (x - O1);
    else if (x < O3) { w = a.w2 + (x - O2); wb = a.w2b + (x - O2); }
    else if (x < O4) w = a.b2 + (x - O3);
    else if (x < O5) { w = a.w3 + (x - O4); wb = a.w3b + (x - O4); }
    else w = a.b3;
    const float m = a.beta1 * a.m[x] + (1.f - a.beta1) * g;
    const float v = a.beta2 * a.v[x] + (1.f - a.beta2) * g * g;
    a.m[x] = m;
    a.v[x] = v;
    const float nw = *w - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
    *w = nw;
    if (wb) *wb = __float2bfloat16(nw);
}

__global__ void k_select(const pastis_cand *pairs, const float *z, int64_t n, float thr, uint32_t *flags) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) flags[p] = z[p] >= thr ? 1u : 0u;
}

__global__ void k_select_scatter(const pastis_cand *pairs, const uint32_t *flags, const uint32_t *off, int64_t n,
                                 pastis_cand *out) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n && flags[p]) out[off[p]] = pairs[p];
}

}  // namespace

static pastis_status features_qt(pastis_ctx *ctx, const uint8_t *d_qcodes, const int64_t *d_qoffsets,
                                 const uint8_t *d_tcodes, const int64_t *d_toffsets, const pastis_cand *d_pairs,
                                 int64_t n_pairs, const pastis_params *params, void *d_x) {
    if (!ctx || n_pairs < 0) return PASTIS_ERR_INVALID_ARG;
    pastis_status s = check_params(params);
    if (s != PASTIS_OK) return s;
    if (n_pairs == 0) return PASTIS_OK;
    if (!d_qcodes || !d_qoffsets || !d_tcodes || !d_toffsets || !d_pairs || !d_x) return PASTIS_ERR_INVALID_ARG;
    int8_t *dmat;
    PASTIS_WS(dmat, ctx, WS_FLAGS, 1024);
    PASTIS_CUDA_TRY(cudaMemcpyAsync(dmat, params->matrix, 576, cudaMemcpyHostToDevice, ctx->stream));
    prof_begin(ctx, "mlp_features");
    k_pair_features<<<(unsigned)ceil_div64(n_pairs, 256), 256, 0, ctx->stream>>>(
        d_qcodes, d_qoffsets, d_tcodes, d_toffsets, d_pairs, n_pairs, params->k, dmat, (__nv_bfloat16 *)d_x);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    return PASTIS_OK;
}

extern "C" pastis_status pastis_pair_features(pastis_ctx *ctx, const uint8_t *d_codes, const int64_t *d_offsets,
                                              const pastis_cand *d_pairs, int64_t n_pairs, const pastis_params *params,
                                              void *d_x) {
    return features_qt(ctx, d_codes, d_offsets, d_codes, d_offsets, d_pairs, n_pairs, params, d_x);
}

extern "C" pastis_status pastis_pair_features_qt(pastis_ctx *ctx, const uint8_t *d_qcodes,
                                                 const int64_t *d_qoffsets, const uint8_t *d_tcodes,
                                                 const int64_t *d_toffsets, const pastis_cand *d_pairs,
                                                 int64_t n_pairs, const pastis_params *params, void *d_x) {
    return features_qt(ctx, d_qcodes, d_qoffsets, d_tcodes, d_toffsets, d_pairs, n_pairs, params, d_x);
}

static mlp_w mlp_weights(const pastis_mlp *net) {
    return mlp_w{(const __nv_bfloat16 *)net->w1b, (const __nv_bfloat16 *)net->w2b, (const __nv_bfloat16 *)net->w3b,
                 net->b1, net->b2, net->b3};
}

cudaError_t mlp_set_smem_limit() {
    cudaError_t e = cudaFuncSetAttribute(k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MLP_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MLP_SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WG_SMEM);
    return e;
}

extern "C" pastis_status pastis_mlp_forward(pastis_ctx *ctx, const pastis_mlp *net, const void *d_x, int64_t n,
                                            float *d_logits) {
    if (!ctx || !net || n < 0 || n > (1 << 30)) return PASTIS_ERR_INVALID_ARG;
    if (n == 0) return PASTIS_OK;
    if (!d_x || !d_logits) return PASTIS_ERR_INVALID_ARG;
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div64(n, TM), ctx->sm_count);
    prof_begin(ctx, "mlp_forward");
    k_mlp<false><<<grid, MLP_THREADS, MLP_SMEM, ctx->stream>>>(mlp_weights(net), (const __nv_bfloat16 *)d_x, n, d_logits,
                                                               mlp_train_io{});
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    return PASTIS_OK;
}

extern "C" pastis_status pastis_mlp_train_step(pastis_ctx *ctx, pastis_mlp *net, const void *d_x, const float *d_y,
                                               int64_t n, float lr, float pos_weight, float *d_loss) {
    if (!ctx || !net || n <= 0 || n > (1 << 22) || !d_x || !d_y) return PASTIS_ERR_INVALID_ARG;
    cudaStream_t st = ctx->stream;
    // scratch: h1, dh1 and dh2 (bf16 n x 256), dz and the loss terms, the partial sums of the gradients
    const int slots = (int)std::min<int64_t>(ceil_div64(n, TM), MLP_SLOTS), grid = std::min(slots, ctx->sm_count);
    const size_t act = (size_t)n * HID * 2, zb = ((size_t)n * 4 + 255) & ~(size_t)255;
    const size_t pb = ((size_t)slots * PART * 4 + 255) & ~(size_t)255;
    char *b;
    PASTIS_WS(b, ctx, WS_MLP, 3 * act + 2 * zb + pb);
    mlp_train_io tr;
    tr.y = d_y;
    tr.pos_weight = pos_weight;
    tr.h1 = (__nv_bfloat16 *)b;
    tr.dh1 = (__nv_bfloat16 *)(b + act);
    tr.dh2 = (__nv_bfloat16 *)(b + 2 * act);
    tr.dz = (float *)(b + 3 * act);
    tr.lrow = (float *)(b + 3 * act + zb);
    tr.part = (float *)(b + 3 * act + 2 * zb);
    tr.slots = slots;
    prof_begin(ctx, "mlp_train");
    k_mlp<true><<<grid, MLP_THREADS, MLP_SMEM, st>>>(mlp_weights(net), (const __nv_bfloat16 *)d_x, n, nullptr, tr);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    prof_begin(ctx, "mlp_wgrad");
    k_mlp_wgrad<<<WG_CTAS, WG_THREADS, WG_SMEM, st>>>((const __nv_bfloat16 *)d_x, tr.h1, tr.dh1, tr.dh2, n, tr.dz,
                                                     tr.lrow, net->grad, net->grad + FEAT * HID + HID,
                                                     net->grad + FEAT * HID + HID * HID + 3 * HID, d_loss);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    net->step += 1;
    adam_args a;
    a.w1 = net->w1; a.b1 = net->b1; a.w2 = net->w2; a.b2 = net->b2; a.w3 = net->w3; a.b3 = net->b3;
    a.w1b = (__nv_bfloat16 *)net->w1b; a.w2b = (__nv_bfloat16 *)net->w2b; a.w3b = (__nv_bfloat16 *)net->w3b;
    a.grad = net->grad; a.m = net->adam_m; a.v = net->adam_v;
    a.lr = lr; a.beta1 = 0.9f; a.beta2 = 0.999f; a.eps = 1e-8f;
    a.c1 = 1.f - powf(a.beta1, (float)net->step);
    a.c2 = 1.f - powf(a.beta2, (float)net->step);
    const int np = FEAT * HID + HID * HID + 3 * HID + 1;
    prof_begin(ctx, "mlp_adam");
    k_mlp_adam<<<(unsigned)((np + 255) / 256), 256, 0, st>>>(a, tr.part, slots);
    PASTIS_LAUNCHED(ctx);
    prof_end(ctx);
    return PASTIS_OK;
}

extern "C" pastis_status pastis_prefilter_select(pastis_ctx *ctx, const pastis_cand *d_pairs, const float *d_logits,
                                                 int64_t n_pairs, float threshold, pastis_cand *d_out,
                                                 int64_t capacity, int64_t *n_out) {
    if (!ctx || !n_out || n_pairs < 0 || capacity < 0) return PASTIS_ERR_INVALID_ARG;
    *n_out = 0;
    if (n_pairs == 0) return PASTIS_OK;
    if (!d_pairs || !d_logits) return PASTIS_ERR_INVALID_ARG;
    if (n_pairs > 0xFFFFFFFFll) return PASTIS_ERR_UNSUPPORTED;
    cudaStream_t st = ctx->stream;
    uint32_t *flags;
    PASTIS_WS(flags, ctx, WS_FILT_FLAGS, sizeof(uint32_t) * (2 * (size_t)n_pairs + 2) + 16);
    uint32_t *off = flags + n_pairs + 1;
    k_select<<<(unsigned)ceil_div64(n_pairs, 256), 256, 0, st>>>(d_pairs, d_logits, n_pairs, threshold, flags);
    PASTIS_LAUNCHED(ctx);
    pastis_status s = exclusive_scan_u32(ctx, flags, off, n_pairs);
    if (s != PASTIS_OK) return s;
    uint32_t total = 0;
    PASTIS_CUDA_TRY(cudaMemcpyAsync(&total, off + n_pairs, sizeof(uint32_t), cudaMemcpyDeviceToHost, st));
    PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    *n_out = total;
    if (capacity < (int64_t)total) return PASTIS_ERR_CAPACITY;
    if (total == 0) return PASTIS_OK;
    if (!d_out) return PASTIS_ERR_INVALID_ARG;
    k_select_scatter<<<(unsigned)ceil_div64(n_pairs, 256), 256, 0, st>>>(d_pairs, flags, off, n_pairs, d_out);
    PASTIS_LAUNCHED(ctx);
    PASTIS_CUDA_TRY(cudaStreamSynchronize(st));
    return PASTIS_OK;
}
