// Cost-model network (config selection of the contraction steps): an MLP
// with two hidden ReLU layers of TN_MLP_HIDDEN units over TN_MLP_IN step
// features, one output (predicted log2 of a step's time per pass).
//
//   z1 = W1 x + b1,  a1 = relu(z1)
//   z2 = W2 a1 + b2, a2 = relu(z2)
//   y  = w3 . a2 + b3
//
// Parameters are one flat FP32 array: W1 [H][D] (row j = hidden unit j),
// b1 [H], W2 [H][H] (row j = unit j of the second layer), b2 [H], w3 [H],
// b3 [1].  Training minimises L = (1/n) sum_i (y_i - t_i)^2.
//
// Kernels:
//   k_mlp_pass<TRAIN>  forward (and, when training, backward) over a
//                      contiguous chunk of rows per CTA, 32 rows at a time;
//                      per-CTA gradient partials go to caller scratch.
//   k_mlp_reduce       sums the partials over CTAs in a fixed order
//                      (deterministic gradients and loss).
//   k_mlp_adam         Adam update (Kingma & Ba, bias-corrected moments).
//   k_mlp_f16          inference with FP16 weights and activations on the
//                      tensor cores, sums in FP32.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "../../include/tn.h"

namespace {

constexpr int D = TN_MLP_IN;
constexpr int H = TN_MLP_HIDDEN;
constexpr int NP = TN_MLP_NPARAMS;
constexpr int OFF_W1 = 0, OFF_B1 = H * D, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H, OFF_W3 = OFF_B2 + H,
              OFF_B3 = OFF_W3 + H;
static_assert(OFF_B3 + 1 == NP, "parameter layout");
constexpr int MAX_CTAS = 152;  // one per SM
constexpr int TR = 32;         // rows per tile
constexpr int WARPS = 8, THREADS = 32 * WARPS;
constexpr int RW = TR / WARPS;  // rows per warp and tile

// Shared memory (floats).  Row strides are 4 mod 32, so that the 16-byte
// reads of eight lanes on consecutive rows touch every bank once.
constexpr int LH = H + 4, LD = D + 4;
constexpr int S_W2 = 0, S_W1 = S_W2 + H * LH, S_X = S_W1 + H * LD, S_A1 = S_X + TR * D, S_DZ2 = S_A1 + TR * LH,
              S_DZ1 = S_DZ2 + TR * LH, S_END_FWD = S_DZ2, S_END = S_DZ1 + TR * LH;
static_assert(H == 128 && D % 4 == 0 && RW == 4, "thread tiles");
static_assert(3 * WARPS * H + 2 * WARPS <= S_X, "the last sums reuse the weights' memory");
template <bool TRAIN>
constexpr size_t pass_smem() { return size_t(TRAIN ? S_END : S_END_FWD) * sizeof(float); }

__device__ __forceinline__ void fma4(float &acc, float4 a, float4 b) {
    acc = fmaf(a.x, b.x, acc);
    acc = fmaf(a.y, b.y, acc);
    acc = fmaf(a.z, b.z, acc);
    acc = fmaf(a.w, b.w, acc);
}

__device__ __forceinline__ float4 lds4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Forward and backward of one CTA's rows as small GEMMs on tiles of 32 rows
// with the weights in shared memory, FP32 FMA.  A warp owns four rows of the
// tile, a lane the units lane + 32 c: the products along a row (z1, z2, dA1)
// read four rows and four units 16 bytes at a time (64 FMA for 8 loads, the
// rows' ones broadcasts) and need no block barrier; the products over the
// rows (dW2: 8 x 8 units a thread in registers for the CTA's whole chunk,
// dW1) take one barrier a tile.  Bound by the shared-memory reads of those
// products: 1.8 M multiply-adds a tile, 7 us at the FMA rate.  A step of
// 4096 rows (gradient, reduction, Adam) takes 33 us; one row at a time per
// CTA, five barriers a row, took 180 us.
template <bool TRAIN>
__global__ void __launch_bounds__(THREADS, 1) k_mlp_pass(const float *__restrict__ P, const float *__restrict__ X,
                                                         const float *__restrict__ T, int64_t n, int64_t chunk,
                                                         float *__restrict__ y_out, float *__restrict__ partial) {
    extern __shared__ __align__(16) float sm[];
    float *W2 = sm + S_W2, *W1 = sm + S_W1, *xs = sm + S_X, *A1 = sm + S_A1;
    float *DZ2 = sm + S_DZ2, *DZ1 = sm + S_DZ1;  // training only
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll 16
    for (int e = tid; e < H * H; e += THREADS) W2[(e / H) * LH + e % H] = P[OFF_W2 + e];
#pragma unroll 4
    for (int e = tid; e < H * D; e += THREADS) W1[(e / D) * LD + e % D] = P[OFF_W1 + e];
    float b1[4], b2[4], w3[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        b1[c] = P[OFF_B1 + lane + 32 * c];
        b2[c] = P[OFF_B2 + lane + 32 * c];
        w3[c] = P[OFF_W3 + lane + 32 * c];
    }
    const float b3 = P[OFF_B3];
    // gradients in registers over the chunk: dW2 rows 8 ty .. + 7, columns
    // 4 tx .. + 3 and 64 + 4 tx .. + 3; dW1 row tid mod H, half of its columns;
    // this warp's share of the vectors' at units lane + 32 c (db1: 4 lane + c)
    const int tx = tid & 15, ty = tid >> 4;
    float g2[8][8], g1[D / 2], gb1[4], gb2[4], gw3[4], gb3 = 0.f, loss = 0.f;
    if (TRAIN) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) g2[i][j] = 0.f;
#pragma unroll
        for (int d = 0; d < D / 2; ++d) g1[d] = 0.f;
#pragma unroll
        for (int c = 0; c < 4; ++c) gb1[c] = gb2[c] = gw3[c] = 0.f;
    }
    const float inv = 2.f / float(n);
    const int64_t r0 = int64_t(blockIdx.x) * chunk;
    const int64_t r1 = r0 + chunk < n ? r0 + chunk : n;
    for (int64_t t0 = r0; t0 < r1; t0 += TR) {
        __syncthreads();  // the weights are in place; the last tile's products over rows are done
        const int rows = int(r1 - t0 < TR ? r1 - t0 : int64_t(TR));
        for (int e = tid; e < TR * D; e += THREADS) xs[e] = e < rows * D ? X[t0 * D + e] : 0.f;
        __syncthreads();
        const int rb = RW * warp;  // this warp's rows of the tile
        float z1[RW][4], z2[RW][4];
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                z1[r][c] = b1[c];
                z2[r][c] = b2[c];
            }
#pragma unroll
        for (int k = 0; k < D; k += 4) {
            float4 x[RW];
#pragma unroll
            for (int r = 0; r < RW; ++r) x[r] = lds4(xs + (rb + r) * D + k);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 w = lds4(W1 + (lane + 32 * c) * LD + k);
#pragma unroll
                for (int r = 0; r < RW; ++r) fma4(z1[r][c], x[r], w);
            }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) A1[(rb + r) * LH + lane + 32 * c] = fmaxf(z1[r][c], 0.f);
        __syncwarp();
#pragma unroll 4
        for (int k = 0; k < H; k += 4) {
            float4 a[RW];
#pragma unroll
            for (int r = 0; r < RW; ++r) a[r] = lds4(A1 + (rb + r) * LH + k);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float4 w = lds4(W2 + (lane + 32 * c) * LH + k);
#pragma unroll
                for (int r = 0; r < RW; ++r) fma4(z2[r][c], a[r], w);
            }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            float s = 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) s = fmaf(w3[c], fmaxf(z2[r][c], 0.f), s);
            const float y = b3 + warp_sum(s);
            const bool live = rb + r < rows;
            if (!TRAIN) {
                if (lane == 0 && live) y_out[t0 + rb + r] = y;
                continue;
            }
            const float e = live ? y - T[t0 + rb + r] : 0.f;
            const float dy = inv * e;
            loss = fmaf(e, e, loss);
            gb3 += dy;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                gw3[c] = fmaf(dy, fmaxf(z2[r][c], 0.f), gw3[c]);
                const float dz = z2[r][c] > 0.f ? dy * w3[c] : 0.f;
                gb2[c] += dz;
                DZ2[(rb + r) * LH + lane + 32 * c] = dz;
            }
        }
        if (!TRAIN) continue;
        __syncwarp();
        // dA1 of units 4 lane .. 4 lane + 3
        float da[RW][4];
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) da[r][c] = 0.f;
#pragma unroll 2
        for (int j = 0; j < H; j += 4) {
            float4 w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = lds4(W2 + (j + q) * LH + 4 * lane);
#pragma unroll
            for (int r = 0; r < RW; ++r) {
                const float4 z = lds4(DZ2 + (rb + r) * LH + j);
                const float zq[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    da[r][0] = fmaf(zq[q], w[q].x, da[r][0]);
                    da[r][1] = fmaf(zq[q], w[q].y, da[r][1]);
                    da[r][2] = fmaf(zq[q], w[q].z, da[r][2]);
                    da[r][3] = fmaf(zq[q], w[q].w, da[r][3]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const float4 a = lds4(A1 + (rb + r) * LH + 4 * lane);  // relu(z1): positive where z1 is
            const float aq[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                da[r][c] = aq[c] > 0.f ? da[r][c] : 0.f;
                gb1[c] += da[r][c];
            }
            *reinterpret_cast<float4 *>(DZ1 + (rb + r) * LH + 4 * lane) = make_float4(da[r][0], da[r][1], da[r][2], da[r][3]);
        }
        __syncthreads();
        // rows past the chunk hold zeros in DZ2 and DZ1
#pragma unroll 2
        for (int r = 0; r < TR; ++r) {
            const float4 za = lds4(DZ2 + r * LH + 8 * ty), zb = lds4(DZ2 + r * LH + 8 * ty + 4);
            const float4 aa = lds4(A1 + r * LH + 4 * tx), ab = lds4(A1 + r * LH + 64 + 4 * tx);
            const float z[8] = {za.x, za.y, za.z, za.w, zb.x, zb.y, zb.z, zb.w};
            const float a[8] = {aa.x, aa.y, aa.z, aa.w, ab.x, ab.y, ab.z, ab.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) g2[i][j] = fmaf(z[i], a[j], g2[i][j]);
        }
        const int gj = tid & (H - 1), gd = (tid / H) * (D / 2);
#pragma unroll 2
        for (int r = 0; r < TR; ++r) {
            const float z = DZ1[r * LH + gj];
#pragma unroll
            for (int d = 0; d < D / 2; d += 4) {
                const float4 x = lds4(xs + r * D + gd + d);
                g1[d] = fmaf(z, x.x, g1[d]);
                g1[d + 1] = fmaf(z, x.y, g1[d + 1]);
                g1[d + 2] = fmaf(z, x.z, g1[d + 2]);
                g1[d + 3] = fmaf(z, x.w, g1[d + 3]);
            }
        }
    }
    if (!TRAIN) return;
    float *out = partial + int64_t(blockIdx.x) * (NP + 1);
    {
        const int gj = tid & (H - 1), gd = (tid / H) * (D / 2);
#pragma unroll
        for (int d = 0; d < D / 2; ++d) out[OFF_W1 + gj * D + gd + d] = g1[d];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) out[OFF_W2 + (8 * ty + i) * H + (j < 4 ? 4 * tx + j : 60 + 4 * tx + j)] = g2[i][j];
    // the vectors: the warps' shares through shared memory, added in warp order
    __syncthreads();
    float *v = sm;  // [3][WARPS][H], then [WARPS][2]
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        v[(0 * WARPS + warp) * H + 4 * lane + c] = gb1[c];
        v[(1 * WARPS + warp) * H + lane + 32 * c] = gb2[c];
        v[(2 * WARPS + warp) * H + lane + 32 * c] = gw3[c];
    }
    if (lane == 0) {
        v[3 * WARPS * H + 2 * warp] = gb3;
        v[3 * WARPS * H + 2 * warp + 1] = loss;
    }
    __syncthreads();
    for (int e = tid; e < 3 * H + 2; e += THREADS) {
        float s = 0.f;
        for (int w = 0; w < WARPS; ++w)
            s += e < 3 * H ? v[((e / H) * WARPS + w) * H + e % H] : v[3 * WARPS * H + 2 * w + (e - 3 * H)];
        const int at = e < H ? OFF_B1 + e : (e < 2 * H ? OFF_B2 + e - H : (e < 3 * H ? OFF_W3 + e - 2 * H : OFF_B3 + e - 3 * H));
        out[at] = s;  // OFF_B3 + 1 = NP: the loss
    }
}
static_assert(OFF_B3 + 1 == NP, "the loss follows the last parameter");

// 32 parameters a block (lane), the CTAs' partials dealt to 8 warps, then
// the warps' sums: a fixed order, and 8 loads in flight for each parameter
// (one thread per parameter walking all CTAs waits for each load in turn).
__global__ void __launch_bounds__(256) k_mlp_reduce(const float *__restrict__ partial, int ctas, int64_t n,
                                                    float *__restrict__ grad, float *__restrict__ loss) {
    __shared__ float s_w[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = blockIdx.x * 32 + lane;
    float s = 0.f;
    if (p <= NP) {
#pragma unroll 8
        for (int c = warp; c < ctas; c += 8) s += partial[int64_t(c) * (NP + 1) + p];
    }
    s_w[warp][lane] = s;
    __syncthreads();
    if (warp != 0 || p > NP) return;
    for (int w = 1; w < 8; ++w) s += s_w[w][lane];
    if (p < NP) grad[p] = s;
    else if (loss) *loss = s / float(n);
}

// (1 - beta) and the bias corrections 1 - beta^t come from the host in
// double precision: in FP32, 1 - 0.999f alone is off by 1.3e-5 relative.
__global__ void k_mlp_adam(float *__restrict__ P, const float *__restrict__ G, float *__restrict__ M,
                           float *__restrict__ V, float lr, float b1, float omb1, float b2, float omb2, float eps,
                           float c1, float c2) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= NP) return;
    const float g = G[p];
    const float m = b1 * M[p] + omb1 * g;
    const float v = b2 * V[p] + omb2 * g * g;
    M[p] = m;
    V[p] = v;
    P[p] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

__global__ void k_mlp_to_half(const float *__restrict__ P, __half *__restrict__ Q) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < NP) Q[p] = __float2half_rn(P[p]);
}

// FP16 inference on the tensor cores (mma.sync: 39 k flops a row make a tile
// of a few microseconds, less than a tcgen05 kernel's set-up).  A warp takes
// 32 rows: layer 1's accumulators are layer 2's A fragments as they stand
// (two 8-column tiles make one 16-deep K step), so the activations never
// leave registers; W1 and W2 are read from shared memory, each B fragment
// for two row tiles.  Weights, features and activations are FP16, every sum
// FP32 (before: 8 half2 products summed in FP16 at a time).  104,622 rows
// take 18 us; one row at a time per 128-thread CTA they took 267 us.
constexpr int LH16 = H + 8;  // halves per W2 row: 8 consecutive rows' 16-byte pieces touch every bank once

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
    const __half2 h = __floats2half2_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&h);
}

__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma_1688(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(b0));
}

constexpr int F16_ROWS = 32;  // rows per warp
static_assert(D == 24, "layer 1: one K step of 16 and one of 8");

__global__ void __launch_bounds__(THREADS) k_mlp_f16(const __half *__restrict__ Q, const float *__restrict__ X,
                                                     int64_t n, float *__restrict__ y_out) {
    __shared__ __align__(16) __half W2[H * LH16];
    __shared__ __align__(16) __half W1[H * D];
    __shared__ float sb1[H], sb2[H], sw3[H];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;  // fragment row and column pair
    if ((reinterpret_cast<uintptr_t>(Q) & 15) == 0) {
        static_assert(OFF_W2 % 8 == 0 && OFF_W1 % 8 == 0, "16-byte pieces");
#pragma unroll
        for (int e = tid; e < H * H / 8; e += THREADS)
            *reinterpret_cast<uint4 *>(W2 + (e / (H / 8)) * LH16 + 8 * (e % (H / 8))) =
                *reinterpret_cast<const uint4 *>(Q + OFF_W2 + 8 * e);
        for (int e = tid; e < H * D / 8; e += THREADS)
            *reinterpret_cast<uint4 *>(W1 + 8 * e) = *reinterpret_cast<const uint4 *>(Q + OFF_W1 + 8 * e);
    } else {
        for (int e = tid; e < H * H; e += THREADS) W2[(e / H) * LH16 + e % H] = Q[OFF_W2 + e];
        for (int e = tid; e < H * D; e += THREADS) W1[e] = Q[OFF_W1 + e];
    }
    if (tid < H) {
        sb1[tid] = __half2float(Q[OFF_B1 + tid]);
        sb2[tid] = __half2float(Q[OFF_B2 + tid]);
        sw3[tid] = __half2float(Q[OFF_W3 + tid]);
    }
    const float b3 = __half2float(Q[OFF_B3]);
    __syncthreads();
    for (int64_t r0 = (int64_t(blockIdx.x) * WARPS + warp) * F16_ROWS; r0 < n;
         r0 += int64_t(gridDim.x) * WARPS * F16_ROWS) {
        // features: row tile m, rows g and g + 8; columns 2t, 2t + 1 of each
        // group of 8 (16-deep step: groups 0, 1; 8-deep step: group 2)
        uint32_t x[2][2][3];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t row = r0 + 16 * m + 8 * h + g;
                const float *xr = X + row * D + 2 * t;
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    x[m][h][q] = row < n ? pack_half2(__ldg(xr + 8 * q), __ldg(xr + 8 * q + 1)) : 0u;
            }
        uint32_t a1[2][H / 16][4];  // layer 2's A fragments
#pragma unroll
        for (int j = 0; j < H / 8; ++j) {  // layer 1, units 8 j .. 8 j + 7
            const __half *w = W1 + (8 * j + g) * D + 2 * t;
            const uint32_t w0 = *reinterpret_cast<const uint32_t *>(w), w1 = *reinterpret_cast<const uint32_t *>(w + 8),
                           w2 = *reinterpret_cast<const uint32_t *>(w + 16);
            const float bl = sb1[8 * j + 2 * t], bh = sb1[8 * j + 2 * t + 1];
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                float c[4] = {bl, bh, bl, bh};
                const uint32_t a[4] = {x[m][0][0], x[m][1][0], x[m][0][1], x[m][1][1]};
                mma_16816(c, a, w0, w1);
                mma_1688(c, x[m][0][2], x[m][1][2], w2);
                a1[m][j / 2][2 * (j & 1)] = pack_half2(fmaxf(c[0], 0.f), fmaxf(c[1], 0.f));
                a1[m][j / 2][2 * (j & 1) + 1] = pack_half2(fmaxf(c[2], 0.f), fmaxf(c[3], 0.f));
            }
        }
        float s[2][2] = {{0.f, 0.f}, {0.f, 0.f}};  // y of rows g, g + 8: this lane's columns
#pragma unroll 4
        for (int j = 0; j < H / 8; ++j) {  // layer 2, units 8 j .. 8 j + 7
            const __half *w = W2 + (8 * j + g) * LH16 + 2 * t;
            const float bl = sb2[8 * j + 2 * t], bh = sb2[8 * j + 2 * t + 1];
            float c[2][4] = {{bl, bh, bl, bh}, {bl, bh, bl, bh}};
#pragma unroll
            for (int k = 0; k < H / 16; ++k) {
                const uint32_t b0 = *reinterpret_cast<const uint32_t *>(w + 16 * k),
                               b1 = *reinterpret_cast<const uint32_t *>(w + 16 * k + 8);
                mma_16816(c[0], a1[0][k], b0, b1);
                mma_16816(c[1], a1[1][k], b0, b1);
            }
            const float wl = sw3[8 * j + 2 * t], wh = sw3[8 * j + 2 * t + 1];
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float2 a2 = __half22float2(__floats2half2_rn(fmaxf(c[m][2 * h], 0.f), fmaxf(c[m][2 * h + 1], 0.f)));
                    s[m][h] = fmaf(wl, a2.x, s[m][h]);
                    s[m][h] = fmaf(wh, a2.y, s[m][h]);
                }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                s[m][h] += __shfl_xor_sync(0xffffffffu, s[m][h], 1);
                s[m][h] += __shfl_xor_sync(0xffffffffu, s[m][h], 2);
                const int64_t row = r0 + 16 * m + 8 * h + g;
                if (t == 0 && row < n) y_out[row] = b3 + s[m][h];
            }
    }
}

int ctas_for(int64_t n) {
    int64_t c = (n + 31) / 32;
    return int(c < 1 ? 1 : (c > MAX_CTAS ? MAX_CTAS : c));
}

}  // namespace

namespace tnk {

size_t mlp_grad_scratch_bytes(int64_t n) { return size_t(ctas_for(n)) * (NP + 1) * sizeof(float); }

cudaError_t mlp_forward(const float *params, const float *X, int64_t n, float *y, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_mlp_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pass_smem<false>());
    if (e != cudaSuccess) return e;
    const int ctas = ctas_for(n);
    const int64_t chunk = (n + ctas - 1) / ctas;
    k_mlp_pass<false><<<ctas, THREADS, pass_smem<false>(), st>>>(params, X, nullptr, n, chunk, y, nullptr);
    return cudaGetLastError();
}

cudaError_t mlp_grad(const float *params, const float *X, const float *t, int64_t n, float *grad, float *loss,
                     float *scratch, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(k_mlp_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pass_smem<true>());
    if (e != cudaSuccess) return e;
    const int ctas = ctas_for(n);
    const int64_t chunk = (n + ctas - 1) / ctas;
    k_mlp_pass<true><<<ctas, THREADS, pass_smem<true>(), st>>>(params, X, t, n, chunk, nullptr, scratch);
    k_mlp_reduce<<<(NP + 1 + 31) / 32, 256, 0, st>>>(scratch, ctas, n, grad, loss);
    return cudaGetLastError();
}

cudaError_t mlp_adam(float *params, const float *grad, float *m, float *v, int32_t step, float lr, float beta1,
                     float beta2, float eps, cudaStream_t st) {
    const double b1 = beta1, b2 = beta2;
    const float c1 = float(1.0 - std::pow(b1, double(step))), c2 = float(1.0 - std::pow(b2, double(step)));
    k_mlp_adam<<<(NP + 255) / 256, 256, 0, st>>>(params, grad, m, v, lr, beta1, float(1.0 - b1), beta2,
                                                 float(1.0 - b2), eps, c1, c2);
    return cudaGetLastError();
}

cudaError_t mlp_to_half(const float *params, uint16_t *params16, cudaStream_t st) {
    k_mlp_to_half<<<(NP + 255) / 256, 256, 0, st>>>(params, reinterpret_cast<__half *>(params16));
    return cudaGetLastError();
}

cudaError_t mlp_forward_f16(const uint16_t *params16, const float *X, int64_t n, float *y, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    const int64_t want = (n + WARPS * F16_ROWS - 1) / (WARPS * F16_ROWS);
    const int ctas = int(want < 2 * MAX_CTAS ? want : 2 * MAX_CTAS);
    k_mlp_f16<<<ctas, THREADS, 0, st>>>(reinterpret_cast<const __half *>(params16), X, n, y);
    return cudaGetLastError();
}

}  // namespace tnk
