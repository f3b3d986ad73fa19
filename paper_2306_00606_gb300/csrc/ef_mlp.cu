// The regression network of the learned ranking path: 16-64-64-1 with ReLU
// on standardised node features, trained with a mean-squared-error loss on
// exact EF by Adam (Kingma and Ba, Algorithm 1).
//
// Every matrix product runs on the tensor cores as BF16 mma.sync m16n8k16
// with FP32 accumulation:
// - inference and the training forward pass take 16 rows per warp;
// - the backward pass computes the data gradients per tile in the same
//   registers;
// - the weight gradients are accumulated by the block over its rows, from
//   shared memory (k_mlp_grad).
// The work is tiny next to the exact EF pass (5.3k parameters): inference
// reads 64 bytes of features per node and is bound by HBM, so the
// warp-level BF16 instructions suffice here (tcgen05 would not pay).
//
// Fragment layouts of m16n8k16 (g = lane / 4, t = lane % 4):
// - A 16x16 row-major: {A[g][2t..2t+1]}, {A[g+8][2t..]}, {A[g][2t+8..]},
//   {A[g+8][2t+8..]};
// - B 16x8: {B[2t..2t+1][g]}, {B[2t+8..2t+9][g]};
// - C 16x8: c0,c1 = C[g][2t..2t+1], c2,c3 = C[g+8][2t..2t+1].
// Two adjacent C tiles of a layer form the A fragment of the next layer's
// 16-wide k-chunk.
#include "ef_internal.cuh"

#include <cuda_bf16.h>

namespace ef {

__device__ __forceinline__ float bf16_to_float(uint16_t u) { return __uint_as_float((uint32_t)u << 16); }

__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The model as one CTA holds it in shared memory.  Weight rows are padded
// (16 -> 24 and 64 -> 72 elements) so that the eight row groups of a
// fragment load fall in different banks (unpadded, 64-element rows put them
// all in one bank: an 8-way conflict that made inference bound by shared
// memory).
constexpr int W1S = 24, W2S = 72;

struct MlpSmem {
    __align__(16) uint16_t w1t[MLP_H * W1S];
    __align__(16) uint16_t w2t[MLP_H * W2S];
    __align__(16) uint16_t w2r[MLP_H * W2S];
    float b1[MLP_H], b2[MLP_H], w3[MLP_H], mean[MLP_F], istd[MLP_F];
    float b3;
};

__device__ void load_model(const ModelDev *M, MlpSmem &s, bool with_w2r) {
    // 16-byte chunks: 2 per W1 row, 8 per W2 row
    const uint4 *src1 = reinterpret_cast<const uint4 *>(M->w1t);
    const uint4 *src2 = reinterpret_cast<const uint4 *>(M->w2t);
    const uint4 *src3 = reinterpret_cast<const uint4 *>(M->w2r);
    for (int i = threadIdx.x; i < MLP_H * 2; i += blockDim.x)
        reinterpret_cast<uint4 *>(s.w1t + (i >> 1) * W1S)[i & 1] = src1[i];
    for (int i = threadIdx.x; i < MLP_H * 8; i += blockDim.x) {
        reinterpret_cast<uint4 *>(s.w2t + (i >> 3) * W2S)[i & 7] = src2[i];
        if (with_w2r) reinterpret_cast<uint4 *>(s.w2r + (i >> 3) * W2S)[i & 7] = src3[i];
    }
    for (int i = threadIdx.x; i < MLP_H; i += blockDim.x) {
        s.b1[i] = M->p[P_B1 + i];
        s.b2[i] = M->p[P_B2 + i];
        s.w3[i] = M->p[P_W3 + i];
    }
    for (int i = threadIdx.x; i < MLP_F; i += blockDim.x) {
        s.mean[i] = M->mean[i];
        s.istd[i] = 1.0f / M->stdv[i];
    }
    if (threadIdx.x == 0) s.b3 = M->p[P_B3];
}

// Forward pass of one 16-row tile.  Rows g and g+8 of this thread are the
// feature rows xg, xg8 (nullptr: a padding row, all zero).
struct Tile {
    uint32_t a1[4];       // standardised features as the layer-1 A fragment
    float h1[8][4];       // layer-1 activations (C tiles)
    float h2[8][4];       // layer-2 activations
    float p0, p1;         // predictions of rows g and g+8 (all four lanes of a group)
};

// The four features a thread needs of one row (2t, 2t+1, 2t+8, 2t+9).
struct RowPart {
    float2 lo, hi;
};

__device__ __forceinline__ RowPart load_row(const float *x) {
    const int t = threadIdx.x & 3;
    if (!x) return RowPart{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    return RowPart{__ldg(reinterpret_cast<const float2 *>(x + 2 * t)),
                   __ldg(reinterpret_cast<const float2 *>(x + 2 * t + 8))};
}

__device__ __forceinline__ void tile_forward(const MlpSmem &s, RowPart rg, RowPart rg8, bool vg, bool vg8, Tile &T);
__device__ __forceinline__ void tile_layers(const MlpSmem &s, Tile &T);

__device__ __forceinline__ void tile_forward(const MlpSmem &s, RowPart rg, RowPart rg8, bool vg, bool vg8, Tile &T) {
    const int t = threadIdx.x & 3;
    const int f0 = 2 * t, f1 = 2 * t + 8;
    float z[2][4];
#pragma unroll
    for (int rr = 0; rr < 2; ++rr) {
        const RowPart &p = rr ? rg8 : rg;
        const bool v = rr ? vg8 : vg;
        z[rr][0] = v ? (p.lo.x - s.mean[f0]) * s.istd[f0] : 0.f;
        z[rr][1] = v ? (p.lo.y - s.mean[f0 + 1]) * s.istd[f0 + 1] : 0.f;
        z[rr][2] = v ? (p.hi.x - s.mean[f1]) * s.istd[f1] : 0.f;
        z[rr][3] = v ? (p.hi.y - s.mean[f1 + 1]) * s.istd[f1 + 1] : 0.f;
    }
    T.a1[0] = pack_bf16(z[0][0], z[0][1]);
    T.a1[1] = pack_bf16(z[1][0], z[1][1]);
    T.a1[2] = pack_bf16(z[0][2], z[0][3]);
    T.a1[3] = pack_bf16(z[1][2], z[1][3]);
    tile_layers(s, T);
}

// Layers 1-3 of a tile whose first-layer operand T.a1 is set.
__device__ __forceinline__ void tile_layers(const MlpSmem &s, Tile &T) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int n = 8 * j + g;
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma16816(c, T.a1, *reinterpret_cast<const uint32_t *>(&s.w1t[n * W1S + 2 * t]),
                 *reinterpret_cast<const uint32_t *>(&s.w1t[n * W1S + 2 * t + 8]));
        const float bb0 = s.b1[8 * j + 2 * t], bb1 = s.b1[8 * j + 2 * t + 1];
        T.h1[j][0] = fmaxf(c[0] + bb0, 0.f);
        T.h1[j][1] = fmaxf(c[1] + bb1, 0.f);
        T.h1[j][2] = fmaxf(c[2] + bb0, 0.f);
        T.h1[j][3] = fmaxf(c[3] + bb1, 0.f);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) T.h2[j][0] = T.h2[j][1] = T.h2[j][2] = T.h2[j][3] = 0.f;
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
        const uint32_t a[4] = {pack_bf16(T.h1[2 * kc][0], T.h1[2 * kc][1]), pack_bf16(T.h1[2 * kc][2], T.h1[2 * kc][3]),
                               pack_bf16(T.h1[2 * kc + 1][0], T.h1[2 * kc + 1][1]),
                               pack_bf16(T.h1[2 * kc + 1][2], T.h1[2 * kc + 1][3])};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int n = 8 * j + g;
            mma16816(T.h2[j], a, *reinterpret_cast<const uint32_t *>(&s.w2t[n * W2S + 16 * kc + 2 * t]),
                     *reinterpret_cast<const uint32_t *>(&s.w2t[n * W2S + 16 * kc + 2 * t + 8]));
        }
    }
    float p0 = 0.f, p1 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int c0 = 8 * j + 2 * t;
        const float bb0 = s.b2[c0], bb1 = s.b2[c0 + 1];
        T.h2[j][0] = fmaxf(T.h2[j][0] + bb0, 0.f);
        T.h2[j][1] = fmaxf(T.h2[j][1] + bb1, 0.f);
        T.h2[j][2] = fmaxf(T.h2[j][2] + bb0, 0.f);
        T.h2[j][3] = fmaxf(T.h2[j][3] + bb1, 0.f);
        p0 += T.h2[j][0] * s.w3[c0] + T.h2[j][1] * s.w3[c0 + 1];
        p1 += T.h2[j][2] * s.w3[c0] + T.h2[j][3] * s.w3[c0 + 1];
    }
    p0 += __shfl_xor_sync(FULL, p0, 1);
    p0 += __shfl_xor_sync(FULL, p0, 2);
    p1 += __shfl_xor_sync(FULL, p1, 1);
    p1 += __shfl_xor_sync(FULL, p1, 2);
    T.p0 = p0 + s.b3;
    T.p1 = p1 + s.b3;
}

constexpr int MLP_WARPS = 8;

// ---------------------------------------------------------------- inference
// Two 16-row tiles per warp step share every weight fragment (one 8-byte
// shared-memory load per pair of tiles: a fragment's two words are stored side
// by side, rows padded to 40 words so that a half-warp's loads fall in
// different banks), layer 2 starts from its biases, and a layer-2 column
// tile is consumed as soon as it is complete, so no activation array is kept.
// Bound by the rate of mma.sync and the shared-memory loads together.
// Measured, 8M rows: 344 us with one tile per step and four-byte loads, 246
// so; at 80 registers (three blocks per SM) 278, four tiles 280, the W2
// fragments in registers (12 warps per SM) 276-292.
constexpr int W2ROW = 40;   // words of a W2 row: 4 k-chunks x 4 lanes x 2 words, padded

struct InferSmem {
    uint2 w1[MLP_H * 4];                   // [n][t] of the one k-chunk
    uint2 w2[MLP_H * W2ROW / 2];           // [n][kc][t]
    float2 b1[MLP_H / 2], b2[MLP_H / 2], w3[MLP_H / 2];
    float mean[MLP_F], istd[MLP_F];
    float b3;
};

__device__ __forceinline__ int w1_at(int n, int t) { return n * 4 + t; }

__device__ void load_infer(const ModelDev *M, InferSmem &s) {
    const uint32_t *w1 = reinterpret_cast<const uint32_t *>(M->w1t), *w2 = reinterpret_cast<const uint32_t *>(M->w2t);
    for (int i = threadIdx.x; i < MLP_H * 4; i += MLP_WARPS * 32) {
        const int n = i >> 2, t = i & 3;
        s.w1[w1_at(n, t)] = make_uint2(w1[n * (MLP_F / 2) + t], w1[n * (MLP_F / 2) + t + 4]);
    }
    for (int i = threadIdx.x; i < MLP_H * 16; i += MLP_WARPS * 32) {
        const int n = i >> 4, kc = i >> 2 & 3, t = i & 3;
        const uint32_t *r = w2 + n * (MLP_H / 2) + 8 * kc + t;
        s.w2[n * (W2ROW / 2) + kc * 4 + t] = make_uint2(r[0], r[4]);
    }
    for (int i = threadIdx.x; i < MLP_H / 2; i += blockDim.x) {
        s.b1[i] = make_float2(M->p[P_B1 + 2 * i], M->p[P_B1 + 2 * i + 1]);
        s.b2[i] = make_float2(M->p[P_B2 + 2 * i], M->p[P_B2 + 2 * i + 1]);
        s.w3[i] = make_float2(M->p[P_W3 + 2 * i], M->p[P_W3 + 2 * i + 1]);
    }
    for (int i = threadIdx.x; i < MLP_F; i += blockDim.x) {
        s.mean[i] = M->mean[i];
        s.istd[i] = 1.0f / M->stdv[i];
    }
    if (threadIdx.x == 0) s.b3 = M->p[P_B3];
}

// Predictions of TILES tiles from their first-layer operands: p[u][0] of
// row g, p[u][1] of row g + 8 (all four lanes of a group).
template <int TILES>
__device__ __forceinline__ void infer_tiles(const InferSmem &s, const uint32_t (&a1)[TILES][4],
                                            float (&p)[TILES][2]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    uint32_t a2[TILES][4][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint2 b = s.w1[w1_at(8 * j + g, t)];
        const float2 bias = s.b1[4 * j + t];
#pragma unroll
        for (int u = 0; u < TILES; ++u) {
            // the bias after the products, as in the training pass: another order
            // rounds some activations to another BF16 value
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            mma16816(c, a1[u], b.x, b.y);
            a2[u][j >> 1][2 * (j & 1)] = pack_bf16(fmaxf(c[0] + bias.x, 0.f), fmaxf(c[1] + bias.y, 0.f));
            a2[u][j >> 1][2 * (j & 1) + 1] = pack_bf16(fmaxf(c[2] + bias.x, 0.f), fmaxf(c[3] + bias.y, 0.f));
        }
    }
#pragma unroll
    for (int u = 0; u < TILES; ++u) p[u][0] = p[u][1] = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float2 bias = s.b2[4 * j + t], w3 = s.w3[4 * j + t];
        float c[TILES][4];
#pragma unroll
        for (int u = 0; u < TILES; ++u) {
            c[u][0] = c[u][2] = bias.x;
            c[u][1] = c[u][3] = bias.y;
        }
#pragma unroll
        for (int kc = 0; kc < 4; ++kc) {
            const uint2 b = s.w2[(8 * j + g) * (W2ROW / 2) + kc * 4 + t];
#pragma unroll
            for (int u = 0; u < TILES; ++u) mma16816(c[u], a2[u][kc], b.x, b.y);
        }
#pragma unroll
        for (int u = 0; u < TILES; ++u) {
            p[u][0] = fmaf(fmaxf(c[u][0], 0.f), w3.x, fmaf(fmaxf(c[u][1], 0.f), w3.y, p[u][0]));
            p[u][1] = fmaf(fmaxf(c[u][2], 0.f), w3.x, fmaf(fmaxf(c[u][3], 0.f), w3.y, p[u][1]));
        }
    }
#pragma unroll
    for (int u = 0; u < TILES; ++u)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            p[u][q] += __shfl_xor_sync(FULL, p[u][q], 1);
            p[u][q] += __shfl_xor_sync(FULL, p[u][q], 2);
            p[u][q] += s.b3;
        }
}

// BF: rows already standardised and rounded to BF16 (8 words per row, word q
// holding features 2q and 2q + 1: words t and t + 4 are the fragment as it
// is), else FP32 rows.  The predictions are equal bit for bit.
template <bool BF, int TILES>
__global__ void __launch_bounds__(MLP_WARPS * 32, 2) k_mlp_infer(const ModelDev *__restrict__ M,
                                                              const void *__restrict__ X_, int32_t n,
                                                              float *__restrict__ out) {
    __shared__ InferSmem s;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, w = threadIdx.x >> 5;
    const float *X = static_cast<const float *>(X_);
    const uint32_t *Xb = static_cast<const uint32_t *>(X_);
    const int64_t tiles = ((int64_t)n + 16 * TILES - 1) / (16 * TILES);
    const int64_t step = (int64_t)gridDim.x * MLP_WARPS;
    // rows g and g + 8 of each tile, loaded ahead of their use (the first ones
    // ahead of the weights)
    RowPart x[TILES][2];
    uint32_t xb[TILES][4];
    auto load = [&](int64_t tile) {
#pragma unroll
        for (int u = 0; u < TILES; ++u)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int64_t r = (tile * TILES + u) * 16 + g + 8 * q;
                if constexpr (BF) {
                    xb[u][q] = r < n ? __ldg(Xb + r * (MLP_F / 2) + t) : 0u;
                    xb[u][q + 2] = r < n ? __ldg(Xb + r * (MLP_F / 2) + t + 4) : 0u;
                } else {
                    x[u][q] = load_row(r < n ? X + r * MLP_F : nullptr);
                }
            }
    };
    int64_t tile = (int64_t)blockIdx.x * MLP_WARPS + w;
    load(tile);
    load_infer(M, s);
    __syncthreads();
    const float m0 = s.mean[2 * t], m1 = s.mean[2 * t + 1], m2 = s.mean[2 * t + 8], m3 = s.mean[2 * t + 9];
    const float i0 = s.istd[2 * t], i1 = s.istd[2 * t + 1], i2 = s.istd[2 * t + 8], i3 = s.istd[2 * t + 9];
    for (; tile < tiles; tile += step) {
        uint32_t a1[TILES][4];
#pragma unroll
        for (int u = 0; u < TILES; ++u)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                if constexpr (BF) {
                    a1[u][q] = xb[u][q];
                    a1[u][q + 2] = xb[u][q + 2];
                } else {
                    const RowPart &r = x[u][q];
                    a1[u][q] = pack_bf16((r.lo.x - m0) * i0, (r.lo.y - m1) * i1);
                    a1[u][q + 2] = pack_bf16((r.hi.x - m2) * i2, (r.hi.y - m3) * i3);
                }
            }
        if (tile + step < tiles) load(tile + step);
        float p[TILES][2];
        infer_tiles(s, a1, p);
        if (t == 0) {
#pragma unroll
            for (int u = 0; u < TILES; ++u)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int64_t r = (tile * TILES + u) * 16 + g + 8 * q;
                    if (r < n) out[r] = p[u][q];
                }
        }
    }
}

// Counter-based row sampling: row r of training step `step` (splitmix64).
__device__ __forceinline__ int sample_row(uint64_t seed, int32_t step, int r, int32_t n) {
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * ((uint64_t)(uint32_t)step * 0x100000000ull + (uint32_t)r + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (int)(z % (uint64_t)n);
}

// Zero the gradient and loss; optionally advance the step counter (which
// seeds the row sampling and Adam's bias corrections).
__global__ void k_mlp_zero(ModelDev *M, bool count_step) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P_N; i += gridDim.x * blockDim.x) M->grad[i] = 0.f;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        M->loss_sum = 0.f;
        if (count_step) M->step += 1;
    }
}

// Gradient of a batch in one kernel.  A block takes 128 rows at a time: each
// warp runs the forward and backward pass of a 16-row tile in registers (loss,
// bias and w3 gradients accumulate there in FP32) and leaves the four BF16
// operands of the weight gradients -- Z, H1, dA2, dA1 -- in shared memory;
// then all warps accumulate dW2 = H1^T dA2 (64 x 64) and dW1 = Z^T dA1
// (16 x 64) over the 128 rows, warp w owning dW2 row tile (w & 3) x column
// tiles 4 (w >> 2) .. +3 and dW1 column tile w, with the transposed fragments
// from ldmatrix.  Rows are padded to 72 (24) elements: the eight 16-byte rows
// of an 8 x 8 matrix fall in different banks.
// Before, the operands went through global memory (416 bytes per row written,
// read again element by element): 700 us for 1M rows, 205 now;
// a training step of 8192 rows 47 -> 28 us.  Bound by latency at the 8 warps
// per SM that 239 registers leave.
constexpr int BATCH_TILE = 16 * MLP_WARPS;
constexpr int ZS = 24, HS = 72;

struct TrainSmem {
    MlpSmem m;
    __align__(16) uint16_t z[BATCH_TILE * ZS];
    __align__(16) uint16_t h1[BATCH_TILE * HS], e2[BATCH_TILE * HS], e1[BATCH_TILE * HS];
    float sums[MLP_WARPS][20][32];   // per lane: the weight gradients of earlier chunks
};

// Chunks whose weight gradients the tensor cores' accumulators hold at most:
// those adds truncate, so short chains added up with rounding are the more
// exact ones.
constexpr int GRAD_CHAIN = 4;

// Four 8 x 8 matrices, transposed; lane l gives the address of row l % 8 of matrix l / 8.
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], const uint16_t *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

__global__ void __launch_bounds__(MLP_WARPS * 32, 1) k_mlp_grad(ModelDev *M, const float *__restrict__ X,
                                                                const float *__restrict__ Y, int32_t n,
                                                                int32_t batch, uint64_t seed, bool sample) {
    extern __shared__ __align__(16) unsigned char train_smem[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(train_smem);
    MlpSmem &s = S.m;
    load_model(M, s, true);
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, w = threadIdx.x >> 5;
    const int32_t step = M->step;
    const float inv_b = 1.0f / (float)batch;
    float gw3[8][2] = {}, gb2[8][2] = {}, gb1[8][2] = {};
    float gb3 = 0.f, loss = 0.f;
    float acc2[4][4] = {}, acc1[4] = {};
    const int mi = w & 3, nj0 = (w >> 2) * 4;
    // this lane's row of an ldmatrix: as A (matrices 1, 3 eight columns on, 2, 3 eight rows on), as B the other way
    const int ar = (lane & 7) + (lane >> 4 & 1) * 8, ac = (lane >> 3 & 1) * 8;
    const int br = (lane & 7) + (lane >> 3 & 1) * 8, bc = (lane >> 4 & 1) * 8;
    const int chunks = (int)(((int64_t)batch + BATCH_TILE - 1) / BATCH_TILE);
    // the next chunk's rows are loaded before this chunk's weight gradients
    RowPart x0, x1;
    float y0, y1;
    bool v0, v1;
    auto load = [&](int chunk) {
        const int64_t r0 = (int64_t)chunk * BATCH_TILE + 16 * w + g, r1 = r0 + 8;
        v0 = chunk < chunks && r0 < batch;
        v1 = chunk < chunks && r1 < batch;
        const int64_t i0 = !v0 ? 0 : sample ? sample_row(seed, step, (int)r0, n) : r0;
        const int64_t i1 = !v1 ? 0 : sample ? sample_row(seed, step, (int)r1, n) : r1;
        x0 = load_row(v0 ? X + i0 * MLP_F : nullptr);
        x1 = load_row(v1 ? X + i1 * MLP_F : nullptr);
        y0 = v0 ? Y[i0] : 0.f;
        y1 = v1 ? Y[i1] : 0.f;
    };
    float *sums = &S.sums[w][0][lane];
#pragma unroll
    for (int i = 0; i < 20; ++i) sums[32 * i] = 0.f;
    int chain = 0;
    load(blockIdx.x);
    for (int chunk = blockIdx.x; chunk < chunks; chunk += gridDim.x) {
        uint32_t *z0 = reinterpret_cast<uint32_t *>(S.z + (16 * w + g) * ZS), *z1 = z0 + 8 * ZS / 2;
        uint32_t *h0 = reinterpret_cast<uint32_t *>(S.h1 + (16 * w + g) * HS), *h8 = h0 + 8 * HS / 2;
        uint32_t *d0p = reinterpret_cast<uint32_t *>(S.e2 + (16 * w + g) * HS), *d8p = d0p + 8 * HS / 2;
        uint32_t *f0p = reinterpret_cast<uint32_t *>(S.e1 + (16 * w + g) * HS), *f8p = f0p + 8 * HS / 2;
        uint32_t e2p[8][2];
        uint32_t active = 0;   // bit 4 j + i: h1[j][i] > 0 (BF16 rounds the smallest positive values to 0)
        {
            Tile T;
            tile_forward(s, x0, x1, v0, v1, T);
            const float e0 = v0 ? T.p0 - y0 : 0.f, e1 = v1 ? T.p1 - y1 : 0.f;
            if (t == 0) loss += e0 * e0 + e1 * e1;
            const float d0 = 2.f * e0 * inv_b, d1 = 2.f * e1 * inv_b;
            if (t == 0) gb3 += d0 + d1;
            z0[t] = T.a1[0];
            z1[t] = T.a1[1];
            z0[t + 4] = T.a1[2];
            z1[t + 4] = T.a1[3];
            // layers 3 and 2: dw3, dA2 = d * w3 * [h2 > 0], db2
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c0 = 8 * j + 2 * t;
                gw3[j][0] += d0 * T.h2[j][0] + d1 * T.h2[j][2];
                gw3[j][1] += d0 * T.h2[j][1] + d1 * T.h2[j][3];
                const float a = T.h2[j][0] > 0.f ? d0 * s.w3[c0] : 0.f;
                const float b = T.h2[j][1] > 0.f ? d0 * s.w3[c0 + 1] : 0.f;
                const float c = T.h2[j][2] > 0.f ? d1 * s.w3[c0] : 0.f;
                const float d = T.h2[j][3] > 0.f ? d1 * s.w3[c0 + 1] : 0.f;
                gb2[j][0] += a + c;
                gb2[j][1] += b + d;
                e2p[j][0] = pack_bf16(a, b);
                e2p[j][1] = pack_bf16(c, d);
#pragma unroll
                for (int i = 0; i < 4; ++i) active |= T.h1[j][i] > 0.f ? 1u << (4 * j + i) : 0u;
                h0[4 * j + t] = pack_bf16(T.h1[j][0], T.h1[j][1]);
                h8[4 * j + t] = pack_bf16(T.h1[j][2], T.h1[j][3]);
                d0p[4 * j + t] = e2p[j][0];
                d8p[4 * j + t] = e2p[j][1];
            }
        }
        // layer 1: dA1 = (dA2 W2^T) * [h1 > 0]; B[k = j][n = i] = W2[i][j] = w2r[i][j]
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int nn = 8 * j + g;
            float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kc = 0; kc < 4; ++kc) {
                const uint32_t a[4] = {e2p[2 * kc][0], e2p[2 * kc][1], e2p[2 * kc + 1][0], e2p[2 * kc + 1][1]};
                mma16816(e, a, *reinterpret_cast<const uint32_t *>(&s.w2r[nn * W2S + 16 * kc + 2 * t]),
                         *reinterpret_cast<const uint32_t *>(&s.w2r[nn * W2S + 16 * kc + 2 * t + 8]));
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) e[i] = active >> (4 * j + i) & 1u ? e[i] : 0.f;
            gb1[j][0] += e[0] + e[2];
            gb1[j][1] += e[1] + e[3];
            f0p[4 * j + t] = pack_bf16(e[0], e[1]);
            f8p[4 * j + t] = pack_bf16(e[2], e[3]);
        }
        load(chunk + gridDim.x);
        __syncthreads();
#pragma unroll 2
        for (int rb = 0; rb < BATCH_TILE; rb += 16) {
            uint32_t a[4], b[4];
            ldsm_x4_trans(a, S.h1 + (rb + ar) * HS + 16 * mi + ac);
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                ldsm_x4_trans(b, S.e2 + (rb + br) * HS + 8 * (nj0 + q) + bc);
                mma16816(acc2[q], a, b[0], b[1]);
                mma16816(acc2[q + 1], a, b[2], b[3]);
            }
            ldsm_x4_trans(a, S.z + (rb + ar) * ZS + ac);
            // (matrices 2 and 3 of the second operand repeat 0 and 1: one column tile is needed)
            ldsm_x4_trans(b, S.e1 + (rb + br) * HS + 8 * w);
            mma16816(acc1, a, b[0], b[1]);
        }
        if (++chain == GRAD_CHAIN || chunk + gridDim.x >= chunks) {
            chain = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    sums[32 * (4 * q + i)] += acc2[q][i];
                    acc2[q][i] = 0.f;
                }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                sums[32 * (16 + i)] += acc1[i];
                acc1[i] = 0.f;
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc2[q][i] = sums[32 * (4 * q + i)];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc1[i] = sums[32 * (16 + i)];
    // reduce over the 8 groups (lanes with equal t hold the same columns)
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                gw3[j][q] += __shfl_xor_sync(FULL, gw3[j][q], o);
                gb2[j][q] += __shfl_xor_sync(FULL, gb2[j][q], o);
                gb1[j][q] += __shfl_xor_sync(FULL, gb1[j][q], o);
            }
    if (g == 0) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int c = 8 * j + 2 * t + q;
                atomicAdd(&M->grad[P_W3 + c], gw3[j][q]);
                atomicAdd(&M->grad[P_B2 + c], gb2[j][q]);
                atomicAdd(&M->grad[P_B1 + c], gb1[j][q]);
            }
    }
    gb3 = warp_sum(gb3);
    loss = warp_sum(loss);
    if (lane == 0) {
        atomicAdd(&M->grad[P_B3], gb3);
        atomicAdd(&M->loss_sum, loss);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = 16 * mi + g, c = 8 * (nj0 + q) + 2 * t;
        atomicAdd(&M->grad[P_W2 + i * MLP_H + c], acc2[q][0]);
        atomicAdd(&M->grad[P_W2 + i * MLP_H + c + 1], acc2[q][1]);
        atomicAdd(&M->grad[P_W2 + (i + 8) * MLP_H + c], acc2[q][2]);
        atomicAdd(&M->grad[P_W2 + (i + 8) * MLP_H + c + 1], acc2[q][3]);
    }
    {
        const int f = g, c = 8 * w + 2 * t;
        atomicAdd(&M->grad[P_W1 + f * MLP_H + c], acc1[0]);
        atomicAdd(&M->grad[P_W1 + f * MLP_H + c + 1], acc1[1]);
        atomicAdd(&M->grad[P_W1 + (f + 8) * MLP_H + c], acc1[2]);
        atomicAdd(&M->grad[P_W1 + (f + 8) * MLP_H + c + 1], acc1[3]);
    }
}

// Opt the gradient kernel in to its shared memory on the current device.
int prepare_mlp() {
    return cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem)) ==
                   cudaSuccess
               ? 0
               : -1;
}

// BF16 copies of the weights in the fragment layouts.
__device__ __forceinline__ void pack_param(ModelDev *M, int i) {
    const uint16_t b = __bfloat16_as_ushort(__float2bfloat16_rn(M->p[i]));
    if (i < P_B1) {
        const int f = (i - P_W1) / MLP_H, j = (i - P_W1) % MLP_H;
        M->w1t[j * MLP_F + f] = b;
    } else if (i >= P_W2 && i < P_B2) {
        const int a = (i - P_W2) / MLP_H, j = (i - P_W2) % MLP_H;
        M->w2t[j * MLP_H + a] = b;
        M->w2r[a * MLP_H + j] = b;
    }
}

__global__ void k_model_pack(ModelDev *M) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P_N; i += gridDim.x * blockDim.x) pack_param(M, i);
}

// One Adam step (bias-corrected moments) with step t = M->step >= 1.
__global__ void k_adam(ModelDev *M, float lr) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const int tstep = M->step;
    const float c1 = 1.f - powf(b1, (float)tstep), c2 = 1.f - powf(b2, (float)tstep);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P_N; i += gridDim.x * blockDim.x) {
        const float gr = M->grad[i];
        const float m = b1 * M->m[i] + (1.f - b1) * gr;
        const float v = b2 * M->v[i] + (1.f - b2) * gr * gr;
        M->m[i] = m;
        M->v[i] = v;
        M->p[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
        pack_param(M, i);
    }
}

// Mean and standard deviation of each feature over the rows (FP64 sums).
__global__ void k_feature_sums(const float *__restrict__ X, int32_t n, double *tmp) {
    __shared__ double s[2 * MLP_F];
    if (threadIdx.x < 2 * MLP_F) s[threadIdx.x] = 0.0;
    __syncthreads();
    const int f = threadIdx.x & (MLP_F - 1);
    double a = 0.0, b = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)n * MLP_F;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double x = X[i];   // blockDim and the stride are multiples of 16: column f throughout
        a += x;
        b += x * x;
    }
    atomicAdd(&s[f], a);
    atomicAdd(&s[MLP_F + f], b);
    __syncthreads();
    if (threadIdx.x < 2 * MLP_F) atomicAdd(&tmp[threadIdx.x], s[threadIdx.x]);
}

__global__ void k_feature_stats(const double *tmp, int32_t n, ModelDev *M) {
    const int f = threadIdx.x;
    if (f < MLP_F) {
        const double mu = tmp[f] / n, var = tmp[MLP_F + f] / n - mu * mu;
        const double sd = var > 1e-12 ? sqrt(var) : 1.0;
        M->mean[f] = (float)mu;
        M->stdv[f] = (float)sd;
    }
}

int launch_feature_stats(const float *x, int32_t n, ModelDev *M, double *tmp, cudaStream_t st) {
    if (n <= 0) return -1;
    if (cudaMemsetAsync(tmp, 0, 2 * MLP_F * sizeof(double), st) != cudaSuccess) return -1;
    k_feature_sums<<<256, 256, 0, st>>>(x, n, tmp);
    k_feature_stats<<<1, 32, 0, st>>>(tmp, n, M);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_model_pack(ModelDev *M, cudaStream_t st) {
    k_model_pack<<<(P_N + 255) / 256, 256, 0, st>>>(M);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// Up to one 16-row tile per warp of the chip (two blocks per SM) each warp has
// one tile: below that line a second tile is work for padding, and the
// smallest calls are the latency of one warp step.  A call of a
// few thousand rows: 15.4 us with two tiles, 14.8 with one.
template <bool BF>
static int infer(const ModelDev *M, const void *x, int32_t n, float *out, int num_sms, cudaStream_t st) {
    const int64_t rows = 16 * MLP_WARPS, cap = (int64_t)num_sms * 2, g = ((int64_t)n + rows - 1) / rows;
    if (g <= cap) {
        k_mlp_infer<BF, 1><<<(unsigned)(g < 1 ? 1 : g), MLP_WARPS * 32, 0, st>>>(M, x, n, out);
    } else {
        const int64_t g2 = (g + 1) / 2;
        k_mlp_infer<BF, 2><<<(unsigned)(g2 > cap ? cap : g2), MLP_WARPS * 32, 0, st>>>(M, x, n, out);
    }
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int launch_mlp_infer(const ModelDev *M, const float *x, int32_t n, float *out, int num_sms, cudaStream_t st) {
    return infer<false>(M, x, n, out, num_sms, st);
}

int launch_mlp_infer_bf16(const ModelDev *M, const uint32_t *xb, int32_t n, float *out, int num_sms,
                          cudaStream_t st) {
    return infer<true>(M, xb, n, out, num_sms, st);
}

// One training (or gradient-only) step over `batch` rows: zero, the
// gradient, and (adam) the update.
int launch_mlp_step(ModelDev *M, const float *x, const float *y, int32_t n, int32_t batch, uint64_t seed, bool sample,
                    bool count_step, bool adam, float lr, int num_sms, cudaStream_t st) {
    k_mlp_zero<<<(P_N + 255) / 256, 256, 0, st>>>(M, count_step);
    const int64_t chunks = ((int64_t)batch + BATCH_TILE - 1) / BATCH_TILE;
    k_mlp_grad<<<(unsigned)(chunks < num_sms ? chunks : num_sms), MLP_WARPS * 32, sizeof(TrainSmem), st>>>(
        M, x, y, n, batch, seed, sample);
    if (adam) k_adam<<<(P_N + 255) / 256, 256, 0, st>>>(M, lr);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace ef
