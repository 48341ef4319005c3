// CUDA-core kernels of the contraction path (sm_103a).
//
//   k_fill           leaf instance blocks for one slice batch (the fused gate
//                    tensors with output legs projected on the bitstrings'
//                    values and sliced legs on the slice's values)
//   k_step_row       one pairwise step C = A (x) B with a small B operand
//                    (N <= 16, K*N <= 256), grouped by shared A instance: each
//                    A row is read once and multiplied by every B block of
//                    its group; the bandwidth-bound "high-rank x low-rank"
//                    contraction of SM Sec. V.A
//   k_step_gemm_simt tiled complex GEMM with gathered (bit-permuted) operand
//                    loads, FP32 FMA; the plain FP32 form of big x big steps
//   k_step_narrow    long rows, few columns per A instance
//   k_step_outer     short rows, many columns
//   k_step_skinny    few outputs per instance, long K
//   k_accumulate     amp[p] += sum over the batch's slices of the root
//                    partials times 2^E, complex128, fixed slice order
//                    (first-level slicing, SM Sec. IV.B)
//   k_xeb            FP64 fixed-order reduction of sum |amp|^2 (Eq. fxeb)
//   k_pt_moments     FP64 sums for the Porter-Thomas mixture fit of the
//                    fidelity (density of Eq. fxeb) and the linear XEB's error
//   k_pt_hist        histogram of x = N |amp|^2 (integer counts)
//   k_sample         one completion per correlated batch, drawn with
//                    probability |amp|^2 / sum over the batch (perfect
//                    sample from a batch, main text on Fig. 3(b), SM Sec. II);
//                    k_sample_rows: batches of at most 32 completions
//
// Power-of-two rescaling: every instance, leaves among them, has the largest
// |component| of its entries recorded (as float bits, atomicMax of non-negative
// floats); its consumer multiplies the loaded values by 2^-e, e the
// exponent of that maximum, and adds e to the output's exponent E.  Scaling
// by a power of two is exact, so with and without it the FP32 results of
// these kernels are bitwise the same (barring subnormals).
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace tnk {

namespace {

__device__ __forceinline__ uint32_t absmax_bits(float2 v) {
    return __float_as_uint(fmaxf(fabsf(v.x), fabsf(v.y)));
}

__device__ __forceinline__ void cfma(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

__device__ __forceinline__ int64_t dep(int64_t x, const int8_t *pos, int nbits) {
    int64_t r = 0;
    for (int j = 0; j < nbits; ++j) r |= ((x >> j) & 1) << pos[j];
    return r;
}

// raise the recorded maximum only when it grows (monotone, so the
// unsynchronised read is safe)
// fire-and-forget global max (a reduction, no returned value: the issuing
// thread never waits on memory)
__device__ __forceinline__ void record_max(uint32_t *slot, uint32_t v) {
    asm volatile("red.relaxed.gpu.global.max.u32 [%0], %1;" ::"l"(slot), "r"(v) : "memory");
}

__global__ void k_fill(const FillJobD *__restrict__ jobs, int64_t njobs, const LeafHighD *__restrict__ highs,
                       int64_t batch, float2 *__restrict__ ws) {
    const int64_t job = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (job >= njobs) return;
    const FillJobD J = jobs[job];
    const LeafHighD H = highs[J.leaf_high];
    int64_t src = J.src;
    for (int c = 0; c < H.cnt; ++c) src += ((batch >> H.j[c]) & 1) * int64_t(H.stride[c]);
    uint32_t mx = 0u;
    for (int e = lane; e < J.n; e += 32) {
        const float2 v = ws[src + e];
        ws[J.dst + e] = v;
        mx = max(mx, absmax_bits(v));
    }
    if (J.mx < 0) return;
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) reinterpret_cast<uint32_t *>(ws)[J.mx] = mx;
}

constexpr int ROW_THREADS = 256;
constexpr int ROW_SB = 2048;  // staged B entries (complex) per block: 16 KB
constexpr int ROW_CH = 32;    // most instances staged at once

// Small-rank step (N = 2^NB <= 16, K*N <= 256), grouped: the output
// instances that read one A instance (a group) are computed together, so
// every A row is read once and multiplied by each of the group's B blocks.
// A row's K-contiguous run (rows are affine: A + m*K) is split over
// L = min(8, K/2) lanes holding KL = K/L complex values each in registers,
// loaded 16 bytes at a time; each output's partial products are summed over
// the row's L lanes with xor-shuffles.  R = 32/L rows per warp pass.
//   uniform (M >= 8R): a block = rows_per_block rows of one group; the
//     group's B blocks (column-affine: K*N contiguous complex each) are
//     staged in shared memory, ROW_SB entries at a time; max-|x| words and
//     exponents are recorded once per instance.
//   small instances (M < 8R): a block = rows_per_block consecutive rows of
//     consecutive groups, each row looping over its group's instances; B
//     comes through the L1 cache.  Schedule 1: rows_per_block consecutive
//     (instance, row) pairs, one per lane group, so that the instances of
//     large groups run in parallel.
template <int NB, int KL>
__global__ void __launch_bounds__(ROW_THREADS) k_step_row(const StepDesc d, int rows_per_block, int64_t mblocks) {
    constexpr int N = 1 << NB;
    __shared__ int8_t s_pCm[40];
    __shared__ int64_t s_offCn[N];
    __shared__ int64_t s_mloC[256];
    __shared__ __align__(16) float2 s_B[ROW_SB];
    __shared__ int64_t s_ib[ROW_CH];
    __shared__ int32_t s_e[ROW_CH], s_EC[ROW_CH];
    __shared__ uint32_t s_mx[ROW_CH];
    __shared__ int64_t s_pass_off[16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = 1 << d.kb;
    const int KN = K * N;
    const int mb = d.mb;
    const int64_t M = int64_t(1) << mb;
    const int L = K / KL;  // lanes per row (row_lanes on the host)
    const int R = 32 / L;
    const int sub = lane / L, kl = lane % L;
    const int passes = rows_per_block / (8 * R);
    if (tid < 40) s_pCm[tid] = d.pCm[tid];
    if (tid < N) s_offCn[tid] = dep(tid, d.pCn, NB);
    __syncthreads();
    {
        const int lob = mb < 8 ? mb : 8;
        s_mloC[tid] = dep(tid & ((1 << lob) - 1), s_pCm, lob);
    }
    __syncthreads();

    // this lane's KL values of row m of A instance ia
    auto load_row = [&](float2 (&a)[KL], int64_t ia, int64_t m, bool valid) {
        const float2 *A = d.A + ia * d.sA + (m << d.kb);
        if (KL == 1) {
            a[0] = valid ? __ldg(A) : make_float2(0.f, 0.f);
        } else {
#pragma unroll
            for (int q = 0; q < KL / 2; ++q) {
                const float4 v = valid ? __ldg(reinterpret_cast<const float4 *>(A + 2 * kl + 2 * L * q))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
                a[2 * q] = make_float2(v.x, v.y);
                a[2 * q + 1] = make_float2(v.z, v.w);
            }
        }
    };
    // acc[n] = sum over this lane's k of a[k] B[n*K + k], then summed over
    // the row's L lanes by recursive halving: at xor level o = 1, 2, 4 a lane
    // keeps one half of the outputs it still holds (the upper half when bit o
    // of its lane index is set) and adds its partner's copy of that half;
    // once one output is left, plain xor sums finish.  Afterwards each lane
    // holds max(1, N / L) outputs (n0, n_held below).
    auto row_times_b = [&](float2 (&acc)[N], const float2 (&a)[KL], const float2 *Bj) {
#pragma unroll
        for (int n = 0; n < N; ++n) acc[n] = make_float2(0.f, 0.f);
        if (KL == 1) {
#pragma unroll
            for (int n = 0; n < N; ++n) cfma(acc[n], a[0], Bj[n * K]);
        } else {
#pragma unroll
            for (int q = 0; q < KL / 2; ++q) {
                const int k = 2 * kl + 2 * L * q;
#pragma unroll
                for (int n = 0; n < N; ++n) {
                    const float4 b = *reinterpret_cast<const float4 *>(Bj + n * K + k);
                    cfma(acc[n], a[2 * q], make_float2(b.x, b.y));
                    cfma(acc[n], a[2 * q + 1], make_float2(b.z, b.w));
                }
            }
        }
#pragma unroll
        for (int t = 0; t < 3; ++t) {
            const int o = 1 << t;
            if (o >= L) break;
            constexpr int W0 = N;
            const int width = W0 >> t;  // a constant once unrolled
            if (width > 1) {
                const bool up = (kl & o) != 0;
#pragma unroll
                for (int n = 0; n < N / 2; ++n) {
                    if (n < (width >> 1)) {
                        const int h = width >> 1;
                        const float2 send = up ? acc[n] : acc[n + h];
                        const float2 keep = up ? acc[n + h] : acc[n];
                        acc[n].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, o);
                        acc[n].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, o);
                    }
                }
            } else {
                acc[0].x += __shfl_xor_sync(0xffffffffu, acc[0].x, o);
                acc[0].y += __shfl_xor_sync(0xffffffffu, acc[0].y, o);
            }
        }
    };
    // outputs this lane holds after row_times_b: acc[j] is output n0 + j
    int n0 = 0, n_held = N;
    for (int t = 0; (1 << t) < L && n_held > 1; ++t) {
        n_held >>= 1;
        if (kl & (1 << t)) n0 += n_held;
    }
    const bool store_lane = N >= L || kl < N;  // higher lane bits hold copies

    if (M >= 8 * R) {
        const int64_t g = int64_t(blockIdx.x) / mblocks;
        const int64_t m0 = (int64_t(blockIdx.x) - g * mblocks) * rows_per_block;
        const int64_t i0 = d.gfirst[g], cnt = d.gfirst[g + 1] - i0;
        const int64_t ia = d.instab[i0].x;
        const int ea = d.mxA ? exp_of(d.mxA[ia]) : 0;
        const int EAa = d.EA[ia] + ea;
        const int ch_max = min(ROW_CH, ROW_SB / KN);
        for (int64_t c0 = 0; c0 < cnt; c0 += ch_max) {
            const int ch = int(cnt - c0 < ch_max ? cnt - c0 : int64_t(ch_max));
            if (tid < ch) {
                const int64_t ib = d.instab[i0 + c0 + tid].y;
                const int eb = d.mxB ? exp_of(d.mxB[ib]) : 0;
                s_ib[tid] = ib;
                s_e[tid] = ea + eb;
                s_EC[tid] = EAa + d.EB[ib] + eb;
                s_mx[tid] = 0u;
            }
            if (tid < passes) s_pass_off[tid] = dep(int64_t(tid) * 8 * R, s_pCm, mb);
            __syncthreads();
            // B staged with each instance's power-of-two rescale folded in (exact)
            for (int e = tid; e < ch * KN; e += ROW_THREADS) {
                const int j = e / KN;
                const float sc = pow2f(-s_e[j]);
                const float2 b = __ldg(d.B + s_ib[j] * d.sB + (e - j * KN));
                s_B[e] = make_float2(b.x * sc, b.y * sc);
            }
            __syncthreads();
            // row m = m0 + it 8R + (warp R + sub): three disjoint bit ranges,
            // so its C offset is this lane's part plus the pass's part
            const int64_t lane_off = dep(m0 + int64_t(warp) * R + sub, s_pCm, mb);
            // max-|x| per instance: in registers across the passes when the
            // chunk has at most 4 instances, reduced over the warp once
            const bool few = ch <= 4;
            uint32_t mxr[4] = {0u, 0u, 0u, 0u};
            // the next pass's A row is loaded while this pass computes
            float2 a_nx[KL];
            load_row(a_nx, ia, m0 + int64_t(warp) * R + sub, true);
            for (int it = 0; it < passes; ++it) {
                float2 a[KL];
#pragma unroll
                for (int q = 0; q < KL; ++q) a[q] = a_nx[q];
                if (it + 1 < passes) load_row(a_nx, ia, m0 + (int64_t(it + 1) * 8 + warp) * R + sub, true);
                const int64_t offC = lane_off + s_pass_off[it];
                for (int j = 0; j < ch; ++j) {
                    float2 acc[N];
                    row_times_b(acc, a, s_B + j * KN);
                    float2 *C = d.C + (i0 + c0 + j) * d.sC + offC;
                    uint32_t mx = 0;
                    if (store_lane) {
#pragma unroll
                        for (int h = 0; h < N; ++h) {
                            if (h >= n_held) break;
                            C[s_offCn[n0 + h]] = acc[h];
                            mx = max(mx, absmax_bits(acc[h]));
                        }
                    }
                    if (d.mxC) {
                        if (few) {
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                if (q == j) mxr[q] = max(mxr[q], mx);
                        } else {
                            const uint32_t r = __reduce_max_sync(0xffffffffu, mx);
                            if (lane == 0 && r) atomicMax(&s_mx[j], r);
                        }
                    }
                }
            }
            if (d.mxC && few) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (q >= ch) break;
                    const uint32_t r = __reduce_max_sync(0xffffffffu, mxr[q]);
                    if (lane == 0 && r) atomicMax(&s_mx[q], r);
                }
            }
            __syncthreads();
            if (tid < ch) {
                const int64_t i = i0 + c0 + tid;
                if (m0 == 0) d.EC[i] = s_EC[tid];
                if (d.mxC && s_mx[tid]) record_max(d.mxC + i, s_mx[tid]);
            }
            __syncthreads();
        }
    } else if (d.sched == 1) {
        // small instances, schedule 1: one output instance row per lane
        // group (instances of large groups run in parallel; their shared A
        // rows come through the caches)
        const int64_t total = d.nInst << mb;
        for (int it = 0; it < passes; ++it) {
            const int64_t gid = int64_t(blockIdx.x) * rows_per_block + (int64_t(it) * 8 + warp) * R + sub;
            const bool valid = gid < total;
            const int64_t gr = valid ? gid : 0;
            const int64_t i = d.inst0 + (gr >> mb), m = gr & (M - 1);
            const int2 ab = d.instab[i];
            const int ea = d.mxA ? exp_of(d.mxA[ab.x]) : 0;
            const int eb = d.mxB ? exp_of(d.mxB[ab.y]) : 0;
            float2 a[KL];
            load_row(a, ab.x, m, valid);
            float2 acc[N];
            row_times_b(acc, a, d.B + int64_t(ab.y) * d.sB);
            const float sc = pow2f(-(ea + eb));
            uint32_t mx = 0;
            if (valid) {
                float2 *C = d.C + i * d.sC + (mb > 8 ? dep(m >> 8, s_pCm + 8, mb - 8) : 0) + s_mloC[m & 255];
                if (store_lane) {
#pragma unroll
                    for (int h = 0; h < N; ++h) {
                        if (h >= n_held) break;
                        const float2 v = make_float2(acc[h].x * sc, acc[h].y * sc);
                        C[s_offCn[n0 + h]] = v;
                        mx = max(mx, absmax_bits(v));
                    }
                }
                if (m == 0 && kl == 0) d.EC[i] = d.EA[ab.x] + ea + d.EB[ab.y] + eb;
            }
            for (int o = L >> 1; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if (d.mxC && valid && kl == 0 && mx) record_max(d.mxC + i, mx);
        }
    } else {
        const int64_t total = d.n_groups << mb;
        for (int it = 0; it < passes; ++it) {
            const int64_t gid = int64_t(blockIdx.x) * rows_per_block + (int64_t(it) * 8 + warp) * R + sub;
            const bool valid = gid < total;
            const int64_t gr = valid ? gid : 0;
            const int64_t g = gr >> mb, m = gr & (M - 1);
            const int64_t i0 = d.gfirst[g];
            const int cnt = valid ? int(d.gfirst[g + 1] - i0) : 0;
            const int64_t ia = d.instab[i0].x;
            const int ea = d.mxA ? exp_of(d.mxA[ia]) : 0;
            float2 a[KL];
            load_row(a, ia, m, valid);
            const int64_t offC = (mb > 8 ? dep(m >> 8, s_pCm + 8, mb - 8) : 0) + s_mloC[m & 255];
            const int jmax = int(__reduce_max_sync(0xffffffffu, uint32_t(cnt)));  // warp-uniform trip count
            for (int j = 0; j < jmax; ++j) {
                const bool vj = j < cnt;
                const int64_t i = i0 + j;
                const int64_t ib = vj ? d.instab[i].y : 0;
                float2 acc[N];
                row_times_b(acc, a, d.B + ib * d.sB);
                const int eb = vj && d.mxB ? exp_of(d.mxB[ib]) : 0;
                const float sc = pow2f(-(ea + eb));
                uint32_t mx = 0;
                if (vj) {
                    float2 *C = d.C + i * d.sC + offC;
                    if (store_lane) {
#pragma unroll
                        for (int h = 0; h < N; ++h) {
                            if (h >= n_held) break;
                            const float2 v = make_float2(acc[h].x * sc, acc[h].y * sc);
                            C[s_offCn[n0 + h]] = v;
                            mx = max(mx, absmax_bits(v));
                        }
                    }
                    if (m == 0 && kl == 0) d.EC[i] = d.EA[ia] + ea + d.EB[ib] + eb;
                }
                for (int o = L >> 1; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                if (d.mxC && vj && kl == 0 && mx) record_max(d.mxC + i, mx);
            }
        }
    }
}

// Grouped SIMT complex GEMM, FP32 FMA.  One CTA: BM rows of the group's A
// instance times BN columns of the group's concatenated B instances (column
// c -> instance gfirst[g] + c / N, column n = c % N), K in chunks of BK.
// 256 threads, 8 x 4 outputs each (rows tm + 16 x, columns 4 tn + y).
constexpr int GBM = 128, GBN = 64, GBK = 16;

__global__ void __launch_bounds__(256) k_step_gemm_simt(const StepDesc d, int ctiles, int mtiles) {
    __shared__ int8_t s_pAm[40], s_pCm[40];
    __shared__ int64_t s_offA[GBM], s_offC[GBM];
    __shared__ int64_t s_bbase[GBN], s_cbase[GBN];
    __shared__ int32_t s_eb[GBN];
    __shared__ uint32_t s_mx[GBN];
    __shared__ float2 s_A[GBK][GBM + 2];
    __shared__ float2 s_B[GBK][GBN + 2];
    __shared__ int64_t s_ia;
    __shared__ int s_ea;
    const int tid = threadIdx.x;
    const int64_t bid = blockIdx.x;
    // schedule 0: row tiles of a column tile on consecutive blocks (the
    // group's B columns stay in L2); 1: column tiles of a row tile on
    // consecutive blocks (the A rows stay in L2)
    int mt, ct;
    int64_t g;
    if (d.sched == 0) {
        mt = int(bid % mtiles);
        const int64_t rest = bid / mtiles;
        ct = int(rest % ctiles);
        g = rest / ctiles;
    } else {
        ct = int(bid % ctiles);
        const int64_t rest = bid / ctiles;
        mt = int(rest % mtiles);
        g = rest / mtiles;
    }
    const int64_t i0 = d.gfirst[g];
    const int64_t icount = d.gfirst[g + 1] - i0;
    const int N = 1 << d.nb;
    const int64_t M = int64_t(1) << d.mb;
    const int K = 1 << d.kb;
    const int64_t cols = icount * N;
    const int64_t c0 = int64_t(ct) * GBN;
    if (c0 >= cols) return;  // uniform across the block
    const int64_t m0 = int64_t(mt) * GBM;
    if (tid < 40) {
        s_pAm[tid] = d.pAm[tid];
        s_pCm[tid] = d.pCm[tid];
    }
    if (tid == 0) {
        const int64_t sig = i0 / d.nOut, beta = i0 - sig * d.nOut;
        s_ia = int64_t(d.sigA[sig]) * d.nOutA + d.outA[beta];
        s_ea = d.mxA ? exp_of(d.mxA[s_ia]) : 0;
    }
    __syncthreads();
    if (tid < GBM) {
        const int64_t m = m0 + tid;
        s_offA[tid] = m < M ? dep(m, s_pAm, d.mb) : 0;
        s_offC[tid] = m < M ? dep(m, s_pCm, d.mb) : 0;
    } else if (tid < GBM + GBN) {
        const int c = tid - GBM;
        const int64_t gc = c0 + c;
        s_mx[c] = 0;
        if (gc < cols) {
            const int64_t inst = i0 + gc / N;
            const int n = int(gc % N);
            const int64_t sig = inst / d.nOut, beta = inst - sig * d.nOut;
            const int64_t ib = int64_t(d.sigB[sig]) * d.nOutB + d.outB[beta];
            s_bbase[c] = ib * d.sB + dep(n, d.pBn, d.nb);
            s_cbase[c] = inst * d.sC + dep(n, d.pCn, d.nb);
            const int eb = d.mxB ? exp_of(d.mxB[ib]) : 0;
            s_eb[c] = eb;
            if (n == 0 && mt == 0) d.EC[inst] = d.EA[s_ia] + s_ea + d.EB[ib] + eb;
        } else {
            s_bbase[c] = -1;
            s_cbase[c] = -1;
            s_eb[c] = 0;
        }
    }
    __syncthreads();
    const float2 *A = d.A + s_ia * d.sA;
    const int tm = tid & 15, tn = tid >> 4;
    float2 acc[8][4];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = make_float2(0.f, 0.f);
    const int bk = K < GBK ? K : GBK;
    for (int k0 = 0; k0 < K; k0 += bk) {
        for (int e = tid; e < bk * GBM; e += 256) {
            const int kk = e % bk, r = e / bk;
            float2 v = make_float2(0.f, 0.f);
            if (m0 + r < M) v = __ldg(A + s_offA[r] + k0 + kk);
            s_A[kk][r] = v;
        }
        for (int e = tid; e < bk * GBN; e += 256) {
            const int kk = e % bk, c = e / bk;
            float2 v = make_float2(0.f, 0.f);
            if (s_bbase[c] >= 0) v = __ldg(d.B + s_bbase[c] + k0 + kk);
            s_B[kk][c] = v;
        }
        __syncthreads();
        for (int kk = 0; kk < bk; ++kk) {
            float2 a[8], b[4];
#pragma unroll
            for (int x = 0; x < 8; ++x) a[x] = s_A[kk][tm + 16 * x];
#pragma unroll
            for (int y = 0; y < 4; ++y) b[y] = s_B[kk][4 * tn + y];
#pragma unroll
            for (int x = 0; x < 8; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) cfma(acc[x][y], a[x], b[y]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int y = 0; y < 4; ++y) {
        const int c = 4 * tn + y;
        if (s_cbase[c] < 0) continue;
        const float sc = pow2f(-(s_ea + s_eb[c]));
        uint32_t mx = 0;
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const int r = tm + 16 * x;
            if (m0 + r >= M) continue;
            const float2 v = make_float2(acc[x][y].x * sc, acc[x][y].y * sc);
            d.C[s_cbase[c] + s_offC[r]] = v;
            mx = max(mx, absmax_bits(v));
        }
        if (d.mxC) {  // lanes tn*16 .. tn*16+15 share column c: reduce each half-warp first
            const unsigned half = (threadIdx.x & 16) ? 0xffff0000u : 0x0000ffffu;
            const uint32_t r = __reduce_max_sync(half, mx);
            if (tm == 0 && r) atomicMax(&s_mx[c], r);
        }
    }
    if (d.mxC) {
        __syncthreads();
        if (tid < GBN && s_cbase[tid] >= 0) {
            const int64_t inst = i0 + (c0 + tid) / N;
            record_max(d.mxC + inst, s_mx[tid]);
        }
    }
}

// Grouped SIMT complex GEMM, FP32 FMA, K >= 2: the same 128 x 64 tiles
// and block order as k_step_gemm_simt, 128 threads of 8 x 8 complex
// outputs each (rows tm + 16 x, columns 8 tn + y), K in chunks of up to 16
// staged in shared memory by cp.async in two stages, so that a chunk's
// loads run while the previous chunk is multiplied.  Shared memory holds A
// and B K-contiguous per row / column (the operands' own order), rows
// padded to 18 complex (144 bytes) so that the 16-byte reads of eight lanes
// on consecutive rows touch every bank once.
constexpr int SBM = 128, SBN = 64, SBK = 16, SLD = 18;
constexpr size_t SIMT2_SMEM = size_t(2) * (SBM + SBN) * SLD * sizeof(float2);

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void *src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

__global__ void __launch_bounds__(128) k_step_gemm_simt2(const StepDesc d, int ctiles, int mtiles) {
    extern __shared__ __align__(16) float2 s2[];
    __shared__ int64_t s_offC[SBM];
    __shared__ int64_t s_bbase[SBN], s_cbase[SBN];
    __shared__ int32_t s_eb[SBN];
    __shared__ uint32_t s_mx[SBN];
    __shared__ int64_t s_ia;
    __shared__ int s_ea;
    const int tid = threadIdx.x;
    const int64_t bid = blockIdx.x;
    int mt, ct;
    int64_t g;
    if (d.sched == 0) {
        mt = int(bid % mtiles);
        const int64_t rest = bid / mtiles;
        ct = int(rest % ctiles);
        g = rest / ctiles;
    } else {
        ct = int(bid % ctiles);
        const int64_t rest = bid / ctiles;
        mt = int(rest % mtiles);
        g = rest / mtiles;
    }
    const int64_t i0 = d.gfirst[g];
    const int64_t icount = d.gfirst[g + 1] - i0;
    const int N = 1 << d.nb;
    const int64_t M = int64_t(1) << d.mb;
    const int K = 1 << d.kb;
    const int64_t cols = icount * N;
    const int64_t c0 = int64_t(ct) * SBN;
    if (c0 >= cols) return;  // uniform across the block
    const int64_t m0 = int64_t(mt) * SBM;
    if (tid == 0) {
        const int64_t sig = i0 / d.nOut, beta = i0 - sig * d.nOut;
        s_ia = int64_t(d.sigA[sig]) * d.nOutA + d.outA[beta];
        s_ea = d.mxA ? exp_of(d.mxA[s_ia]) : 0;
    }
    __syncthreads();
    {
        const int64_t m = m0 + tid;
        s_offC[tid] = m < M ? dep(m, d.pCm, d.mb) : 0;
    }
    if (tid < SBN) {
        const int c = tid;
        const int64_t gc = c0 + c;
        s_mx[c] = 0;
        if (gc < cols) {
            const int64_t inst = i0 + gc / N;
            const int n = int(gc % N);
            const int64_t sig = inst / d.nOut, beta = inst - sig * d.nOut;
            const int64_t ib = int64_t(d.sigB[sig]) * d.nOutB + d.outB[beta];
            s_bbase[c] = ib * d.sB + (int64_t(n) << d.kb);  // B is K-major and affine
            s_cbase[c] = inst * d.sC + dep(n, d.pCn, d.nb);
            const int eb = d.mxB ? exp_of(d.mxB[ib]) : 0;
            s_eb[c] = eb;
            if (n == 0 && mt == 0) d.EC[inst] = d.EA[s_ia] + s_ea + d.EB[ib] + eb;
        } else {
            s_bbase[c] = -1;
            s_cbase[c] = -1;
            s_eb[c] = 0;
        }
    }
    __syncthreads();
    const float2 *A = d.A + s_ia * d.sA;  // row m at m * K: K-major and affine
    const int bk = K < SBK ? K : SBK;      // complex k per chunk (even: K >= 2)
    const int pieces = bk >> 1;            // 16-byte pieces per row / column and chunk
    const int nchunk = K / bk;
    // stage st: A at s2 + st * SBM * SLD, B at s2 + 2 * SBM * SLD + st * SBN * SLD
    // one chunk's cp.async: piece q of row r at (r, 2q); consecutive threads
    // take consecutive pieces of a row (coalesced)
    auto issue = [&](int ch, int st) {
        const int k0 = ch * bk;
        for (int e = tid; e < SBM * pieces; e += 128) {
            const int r = e / pieces, q = e - r * pieces;
            const bool v = m0 + r < M;
            const float2 *src = v ? A + ((m0 + r) << d.kb) + k0 + 2 * q : A;
            cp_async16_zfill(static_cast<uint32_t>(__cvta_generic_to_shared(s2 + st * SBM * SLD + r * SLD + 2 * q)), src,
                             v);
        }
        for (int e = tid; e < SBN * pieces; e += 128) {
            const int c = e / pieces, q = e - c * pieces;
            const int64_t bb = s_bbase[c];
            const bool v = bb >= 0;
            const float2 *src = v ? d.B + bb + k0 + 2 * q : d.B;
            cp_async16_zfill(
                static_cast<uint32_t>(__cvta_generic_to_shared(s2 + 2 * SBM * SLD + st * SBN * SLD + c * SLD + 2 * q)),
                src, v);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    const int tm = tid & 15, tn = tid >> 4;
    float2 acc[8][8];
#pragma unroll
    for (int x = 0; x < 8; ++x)
#pragma unroll
        for (int y = 0; y < 8; ++y) acc[x][y] = make_float2(0.f, 0.f);
    issue(0, 0);
    for (int ch = 0; ch < nchunk; ++ch) {
        if (ch + 1 < nchunk) {
            issue(ch + 1, (ch + 1) & 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const float2 *a_s = s2 + (ch & 1) * SBM * SLD + tm * SLD;
        const float2 *b_s = s2 + 2 * SBM * SLD + (ch & 1) * SBN * SLD + (8 * tn) * SLD;
        for (int kk = 0; kk < bk; kk += 2) {
            float4 a[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) a[x] = *reinterpret_cast<const float4 *>(a_s + 16 * x * SLD + kk);
#pragma unroll
            for (int y = 0; y < 8; ++y) {
                const float4 b = *reinterpret_cast<const float4 *>(b_s + y * SLD + kk);
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    cfma(acc[x][y], make_float2(a[x].x, a[x].y), make_float2(b.x, b.y));
                    cfma(acc[x][y], make_float2(a[x].z, a[x].w), make_float2(b.z, b.w));
                }
            }
        }
        __syncthreads();  // the stage is refilled two chunks later
    }
#pragma unroll
    for (int y = 0; y < 8; ++y) {
        const int c = 8 * tn + y;
        if (s_cbase[c] < 0) continue;
        const float sc = pow2f(-(s_ea + s_eb[c]));
        uint32_t mx = 0;
#pragma unroll
        for (int x = 0; x < 8; ++x) {
            const int r = tm + 16 * x;
            if (m0 + r >= M) continue;
            const float2 v = make_float2(acc[x][y].x * sc, acc[x][y].y * sc);
            d.C[s_cbase[c] + s_offC[r]] = v;
            mx = max(mx, absmax_bits(v));
        }
        if (d.mxC) {  // lanes tn*16 .. tn*16+15 share column c: reduce each half-warp first
            const unsigned half = (threadIdx.x & 16) ? 0xffff0000u : 0x0000ffffu;
            const uint32_t r = __reduce_max_sync(half, mx);
            if (tm == 0 && r) atomicMax(&s_mx[c], r);
        }
    }
    if (d.mxC) {
        __syncthreads();
        if (tid < SBN && s_cbase[tid] >= 0) {
            const int64_t inst = i0 + (c0 + tid) / N;
            record_max(d.mxC + inst, s_mx[tid]);
        }
    }
}

// Steps with a short row and many columns (K <= 32, N >= 32, M >= 32; reached
// by FP32 steps and, K <= 4, by those that the tensor cores do not take):
// nearly all of their bytes are C's.  A block takes a column tile (64 columns, B in
// shared memory) and 256 RX `passes` rows; a thread holds RX rows of A in
// registers and walks the columns, B's entries as broadcasts, so that a
// warp's 32 rows, neighbours in C where the layout allows, are stored by one
// instruction.  Bound by C's stores, from K = 16 on by the instruction issue
// (67 % of the slots, FMA pipe 52 %) and the shared-memory reads of B.  The GEMM
// kernel stages 16 k a chunk, stores 16 rows an instruction and pads 32
// columns to 64: 7.36 ms for 2^15 x 4 x 32 with 1024 instances (9.7 GB, 1.43
// ms), 1.69 here; 2^10 x 32 x 32 with 8192 (1.1 ms of FMA) and 2^14 x 16 x 32
// with 256 together 5.7, 2.2 here.
// (rlog: log2 of the rows side by side, min(M, 256); the block's other
// threads take other columns.)
template <int KB, int RX>
__global__ void __launch_bounds__(256) k_step_outer(const StepDesc d, int rlog, int passes, int mtiles) {
    constexpr int K = 1 << KB;
    __shared__ __align__(16) float2 s_b[64 * K];
    __shared__ int64_t s_cbase[64];
    __shared__ float s_sc[64];
    __shared__ uint32_t s_mx[64];
    __shared__ int8_t s_pCm[40];
    const int tid = threadIdx.x, lane = tid & 31;
    const int mt = int(blockIdx.x % mtiles);
    // {first instance, count, A instance, first column} of 64 columns
    const int4 rec = __ldg(d.trec + blockIdx.x / mtiles);
    const int N = 1 << d.nb;
    const int ncols = int(min((int64_t(rec.y) << d.nb) - rec.w, int64_t(64)));
    if (tid < 40) s_pCm[tid] = d.pCm[tid];
    if (tid < 64) {
        s_mx[tid] = 0u;
        if (tid < ncols) {
            const int64_t inst = rec.x + ((int64_t(rec.w) + tid) >> d.nb);
            const int n = (rec.w + tid) & (N - 1);
            const int ib = d.instab[inst].y;
            const int ea = d.mxA ? exp_of(d.mxA[rec.z]) : 0, eb = d.mxB ? exp_of(d.mxB[ib]) : 0;
            s_cbase[tid] = inst * d.sC + dep(n, d.pCn, d.nb);
            s_sc[tid] = pow2f(-(ea + eb));
            if (n == 0 && mt == 0) d.EC[inst] = d.EA[rec.z] + ea + d.EB[ib] + eb;
        }
    }
    for (int e = tid; e < ncols * K; e += 256) {
        const int64_t gc = int64_t(rec.w) + (e >> KB);
        const int ib = d.instab[rec.x + (gc >> d.nb)].y;
        s_b[e] = __ldg(d.B + int64_t(ib) * d.sB + ((gc & (N - 1)) << KB) + (e & (K - 1)));
    }
    __syncthreads();
    const int R = 1 << rlog, cw = 64 >> (8 - rlog);
    const int c0 = (tid >> rlog) * cw, c1 = min(c0 + cw, ncols);  // the same for a warp
    const int run = N < 64 ? N - 1 : 63;                          // columns of an instance in the tile, less one
    const float2 *A = d.A + int64_t(rec.z) * d.sA;
    const int64_t m0 = int64_t(mt) * passes * (RX << rlog) + (tid & (R - 1));
    for (int p = 0; p < passes; ++p) {
        float2 a[RX][K];
        float2 *C[RX];
#pragma unroll
        for (int x = 0; x < RX; ++x) {
            const int64_t m = m0 + (int64_t(p * RX + x) << rlog);
            if (KB == 0) {
                a[x][0] = __ldg(A + m);
            } else {
#pragma unroll
                for (int k = 0; k < K; k += 2) {
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(A + (m << KB) + k));
                    a[x][k] = make_float2(v.x, v.y);
                    a[x][k + (KB > 0)] = make_float2(v.z, v.w);
                }
            }
            C[x] = d.C + dep(m, s_pCm, d.mb);
        }
        uint32_t mx = 0u;
        for (int c = c0; c < c1; ++c) {
            float2 acc[RX];
#pragma unroll
            for (int x = 0; x < RX; ++x) acc[x] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float2 b = s_b[(c << KB) + k];
#pragma unroll
                for (int x = 0; x < RX; ++x) cfma(acc[x], a[x][k], b);
            }
            const float sc = s_sc[c];
            const int64_t off = s_cbase[c];
#pragma unroll
            for (int x = 0; x < RX; ++x) {
                const float2 v = make_float2(acc[x].x * sc, acc[x].y * sc);
                C[x][off] = v;
                mx = max(mx, absmax_bits(v));
            }
            if (d.mxC && (((c & run) == run) || c + 1 == c1)) {  // the instance's last column here
                mx = __reduce_max_sync(0xffffffffu, mx);
                if (lane == 0 && mx) atomicMax(&s_mx[c & ~run], mx);
                mx = 0u;
            }
        }
    }
    if (d.mxC) {
        __syncthreads();
        if (tid < ncols && s_mx[tid]) record_max(d.mxC + rec.x + ((int64_t(rec.w) + tid) >> d.nb), s_mx[tid]);
    }
}

// Steps with a long row and few columns per A instance (K >= 32, K N <= 256,
// M >= 128), grouped: a block takes 128 rows of a group's A instance and all
// of the group's concatenated columns (the instances that share it), 8 or 16
// at a time, so A is read once for most groups and from L2 for the others'
// further columns.  Chunks of 8 complex k of A (128 rows x 64 bytes) and B
// arrive by cp.async in three stages; a thread holds 2 or 4 rows x 4 columns,
// rows 32 apart, and reads both operands 16 bytes at a time (64 FMA for 6
// loads or 128 for 8, B's as broadcasts).  Groups of 8 columns on average
// take tiles of 8, on which all four warps work; with tiles of 16 two of them
// would only copy (38.3 against 39.8 ms of the step below).  In tiles of 16
// the four columns of a warp rotate with the block, so that tiles with fewer
// load all four schedulers.  Bound by the instruction issue in tiles of 16 (77 %
// of the slots, FMA pipe 55 %, DRAM 38 % on 2^14 x 64 x 2 with 505 instances on
// 64), in tiles of 8 by its latencies (issue 53 %, DRAM 45 %); a block lives for
// little more than those, so six of them share an SM.  The per-row kernel held a row of 64 in two
// lanes' registers, read B from shared memory for every row and instance
// again and loaded 32 bytes a row at a time: 4.47 ms on 2^8 x 64 x 2 with
// 64448 A instances of 1 to 10 (9.5 GB, 1.40 ms of HBM), 2.40 ms here (1.9
// without the FMAs).
constexpr int NBK = 8, NLD = NBK + 2, NST = 3;

// WR x WC warps, a warp 32 RX rows x 4 columns
template <int WR, int WC, int RX>
struct NarrowTile {
    static constexpr int ROWS = 32 * WR * RX, COLS = 4 * WC, THREADS = 32 * WR * WC;
    static constexpr size_t SMEM = size_t(NST) * (ROWS + COLS) * NLD * sizeof(float2);
};

template <int WR, int WC, int RX, int BLOCKS>
__global__ void __launch_bounds__(32 * WR * WC, BLOCKS) k_step_narrow(const StepDesc d, int mtiles) {
    using T = NarrowTile<WR, WC, RX>;
    constexpr int NBM = T::ROWS, NBN = T::COLS, NT = T::THREADS;
    static_assert(NT >= 40 && NBN * NBK / 2 <= NT, "threads of the set-up");
    extern __shared__ __align__(16) float2 sn[];
    __shared__ int64_t s_bbase[NBN], s_cbase[NBN];
    __shared__ int32_t s_e[NBN];
    __shared__ uint32_t s_mx[NBN];
    __shared__ int8_t s_pCm[40];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t bid = blockIdx.x;
    const int mt = int(bid % mtiles);
    // {first instance, count, A instance, first column} of 64 columns
    const int4 rec = __ldg(d.trec + bid / mtiles);
    const int N = 1 << d.nb, K = 1 << d.kb;
    const int64_t M = int64_t(1) << d.mb;
    const int cend = min(rec.y << d.nb, rec.w + 64);  // columns of the group
    const int64_t m0 = int64_t(mt) * NBM;
    const float2 *A = d.A + int64_t(rec.z) * d.sA + (m0 << d.kb);
    const int nchunk = K / NBK;
    float2 *sa = sn, *sb = sn + NST * NBM * NLD;
    auto issue_a = [&](int ch) {  // 16-byte pieces, four a row (M >= NBM: every row exists)
#pragma unroll
        for (int e = tid; e < NBM * NBK / 2; e += NT) {
            const int r = e >> 2, q = e & 3;
            cp_async16_zfill(static_cast<uint32_t>(__cvta_generic_to_shared(sa + ((ch % NST) * NBM + r) * NLD + 2 * q)),
                             A + (int64_t(r) << d.kb) + ch * NBK + 2 * q, true);
        }
    };
    auto issue_b = [&](int ch) {
        if (tid < NBN * NBK / 2) {
            const int c = tid >> 2, q = tid & 3;
            const bool v = s_bbase[c] >= 0;
            cp_async16_zfill(static_cast<uint32_t>(__cvta_generic_to_shared(sb + ((ch % NST) * NBN + c) * NLD + 2 * q)),
                             v ? d.B + s_bbase[c] + ch * NBK + 2 * q : d.B, v);
        }
    };
    auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };
    if (tid < 40) s_pCm[tid] = d.pCm[tid];
    for (int c0 = rec.w; c0 < cend; c0 += NBN) {  // the same for a block
        if (c0 > rec.w) __syncthreads();  // the stages and the columns' records are reused
        const int ncols = min(cend - c0, NBN);
        issue_a(0);
        issue_a(1);
        if (tid < NBN) {
            s_mx[tid] = 0u;
            s_bbase[tid] = -1;
            if (tid < ncols) {
                const int inst = rec.x + ((c0 + tid) >> d.nb);
                const int n = (c0 + tid) & (N - 1);
                const int ib = d.instab[inst].y;
                const int ea = d.mxA ? exp_of(d.mxA[rec.z]) : 0, eb = d.mxB ? exp_of(d.mxB[ib]) : 0;
                s_bbase[tid] = int64_t(ib) * d.sB + (int64_t(n) << d.kb);
                s_cbase[tid] = int64_t(inst) * d.sC + dep(n, d.pCn, d.nb);
                s_e[tid] = ea + eb;
                if (n == 0 && mt == 0) d.EC[inst] = d.EA[rec.z] + ea + d.EB[ib] + eb;
            }
        }
        __syncthreads();
        issue_b(0);
        commit();
        issue_b(1);
        commit();
        const int cg = WC == 4 ? ((tid >> 5) + int(bid)) & 3 : (tid >> 5) % WC;
        const int r0 = (tid >> 5) / WC * 32 * RX + lane;  // the thread's rows: r0 + 32 x
        const bool works = 4 * cg < ncols;  // the same for a warp
        float2 acc[RX][4];
#pragma unroll
        for (int x = 0; x < RX; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) acc[x][y] = make_float2(0.f, 0.f);
        for (int ch = 0; ch < nchunk; ++ch) {
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncthreads();  // chunk ch is in place; every warp is done with chunk ch - 1
            if (ch + 2 < nchunk) {
                issue_a(ch + 2);
                issue_b(ch + 2);
            }
            commit();
            if (works) {
                const float2 *a_s = sa + ((ch % NST) * NBM + r0) * NLD, *b_s = sb + ((ch % NST) * NBN + 4 * cg) * NLD;
#pragma unroll
                for (int kk = 0; kk < NBK; kk += 2) {
                    float4 a[RX], b[4];
#pragma unroll
                    for (int x = 0; x < RX; ++x) a[x] = *reinterpret_cast<const float4 *>(a_s + 32 * x * NLD + kk);
#pragma unroll
                    for (int y = 0; y < 4; ++y) b[y] = *reinterpret_cast<const float4 *>(b_s + y * NLD + kk);
#pragma unroll
                    for (int x = 0; x < RX; ++x)
#pragma unroll
                        for (int y = 0; y < 4; ++y) {
                            cfma(acc[x][y], make_float2(a[x].x, a[x].y), make_float2(b[y].x, b[y].y));
                            cfma(acc[x][y], make_float2(a[x].z, a[x].w), make_float2(b[y].z, b[y].w));
                        }
                }
            }
        }
        if (works) {
            int64_t off[RX];
#pragma unroll
            for (int x = 0; x < RX; ++x) off[x] = dep(m0 + r0 + 32 * x, s_pCm, d.mb);
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const int c = 4 * cg + y;
                if (c >= ncols) break;  // the same for a warp
                const float sc = pow2f(-s_e[c]);
                float2 *C = d.C + s_cbase[c];
                uint32_t mx = 0u;
#pragma unroll
                for (int x = 0; x < RX; ++x) {
                    const float2 v = make_float2(acc[x][y].x * sc, acc[x][y].y * sc);
                    C[off[x]] = v;
                    mx = max(mx, absmax_bits(v));
                }
                if (d.mxC) {
                    mx = __reduce_max_sync(0xffffffffu, mx);
                    if (lane == 0 && mx) atomicMax(&s_mx[c], mx);
                }
            }
        }
        if (d.mxC) {
            __syncthreads();
            if (tid < ncols && s_mx[tid]) record_max(d.mxC + rec.x + ((c0 + tid) >> d.nb), s_mx[tid]);
        }
    }
}

// Steps with few outputs per instance (M N <= 32, N <= 8) and a long K (the
// root of a plan, with its open qubits, and what is left of the ranks just
// below it).  A unit is one instance and RM of its rows against its N
// columns: its lanes walk the K-contiguous runs side by side, 16 bytes a
// load, each B value used for RM rows and each A value for N columns from
// registers (RM N <= 8 accumulators), then the lanes' sums are added in a
// fixed order.  Bound by HBM: 8 (A + B) bytes per output row.  A GEMM tile
// of 128 x 64 would hold RM N live outputs of 8192 and walk K serially:
// M = 16, K = 2^15, N = 1, 256 instances (1.1 GB, 0.17 ms of HBM) took
// 13.4 ms on the SIMT GEMM, about 0.3 ms here (the contraction that ends in
// it 27.3 -> 14.2 ms).
// W = 8: a block per unit (long K, or too few units to fill the chip with
// warps); W = 1: a warp per unit.
template <int RM, int N, int W>
__global__ void __launch_bounds__(256) k_step_skinny(const StepDesc d, int64_t units) {
    __shared__ float2 s_part[8][RM * N];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t u = W == 8 ? int64_t(blockIdx.x) : int64_t(blockIdx.x) * 8 + warp;
    if (W == 1 && u >= units) return;  // a whole warp
    constexpr int RMB = RM == 1 ? 0 : (RM == 2 ? 1 : (RM == 4 ? 2 : 3));
    const int rbits = d.mb - RMB;  // row blocks per instance (log2)
    const int64_t i = d.inst0 + (u >> rbits);
    const int m0 = int(u & ((int64_t(1) << rbits) - 1)) * RM;
    const int2 ab = d.instab[i];
    const int K2 = 1 << (d.kb - 1);  // 16-byte pieces per row
    const float4 *a4 = reinterpret_cast<const float4 *>(d.A + int64_t(ab.x) * d.sA + (int64_t(m0) << d.kb));
    const float4 *b4 = reinterpret_cast<const float4 *>(d.B + int64_t(ab.y) * d.sB);
    float2 acc[RM][N];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int n = 0; n < N; ++n) acc[r][n] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int q = W == 8 ? tid : lane; q < K2; q += 32 * W) {
        float4 a[RM], b[N];
#pragma unroll
        for (int r = 0; r < RM; ++r) a[r] = __ldg(a4 + int64_t(r) * K2 + q);
#pragma unroll
        for (int n = 0; n < N; ++n) b[n] = __ldg(b4 + int64_t(n) * K2 + q);
#pragma unroll
        for (int r = 0; r < RM; ++r)
#pragma unroll
            for (int n = 0; n < N; ++n) {
                cfma(acc[r][n], make_float2(a[r].x, a[r].y), make_float2(b[n].x, b[n].y));
                cfma(acc[r][n], make_float2(a[r].z, a[r].w), make_float2(b[n].z, b[n].w));
            }
    }
    float2 mine = make_float2(0.f, 0.f);  // lane j < RM N: output (row j / N, column j mod N)
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int n = 0; n < N; ++n) {
            float2 t = acc[r][n];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
                t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
            }
            if (lane == r * N + n) mine = t;
        }
    if (W == 8) {
        if (lane < RM * N) s_part[warp][lane] = mine;
        __syncthreads();
        if (warp != 0) return;
        if (lane < RM * N) {
            mine = s_part[0][lane];
            for (int w = 1; w < 8; ++w) {
                mine.x += s_part[w][lane].x;
                mine.y += s_part[w][lane].y;
            }
        }
    }
    const int ea = d.mxA ? exp_of(d.mxA[ab.x]) : 0;
    const int eb = d.mxB ? exp_of(d.mxB[ab.y]) : 0;
    const float sc = pow2f(-(ea + eb));
    uint32_t mx = 0u;
    if (lane < RM * N) {
        const float2 v = make_float2(mine.x * sc, mine.y * sc);
        d.C[i * d.sC + dep(m0 + lane / N, d.pCm, d.mb) + dep(lane % N, d.pCn, d.nb)] = v;
        mx = absmax_bits(v);
    }
    if (lane == 0 && m0 == 0) d.EC[i] = d.EA[ab.x] + ea + d.EB[ab.y] + eb;
    if (d.mxC) {
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0 && mx) record_max(d.mxC + i, mx);
    }
}

// root entry of completion x: its r bits reversed (root bit t = the t-th
// lowest open qubit; x's most significant bit = the lowest open qubit)
__device__ __forceinline__ int64_t root_entry(int64_t x, int r) {
    return r == 0 ? 0 : int64_t(__brevll(uint64_t(x)) >> (64 - r));
}

// one thread per (input row, completion): amps[p 2^r + x] += the sum over
// the pass's slice instances, in slice order, of root entry x times 2^E
__global__ void k_accumulate(const float2 *__restrict__ root, const int32_t *__restrict__ E,
                             const int32_t *__restrict__ uniq, int64_t k, int64_t n_sig, int32_t n_out, int r,
                             double2 *__restrict__ amps) {
    const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= (k << r)) return;
    const int64_t p = q >> r, x = q & ((int64_t(1) << r) - 1);
    const int64_t beta = uniq[p], j = root_entry(x, r);
    double re = 0.0, im = 0.0;
    for (int64_t s = 0; s < n_sig; ++s) {
        const int64_t idx = s * n_out + beta;
        const float2 v = root[(idx << r) + j];
        const int e = E[idx];
        re += ldexp(double(v.x), e);
        im += ldexp(double(v.y), e);
    }
    double2 a = amps[q];
    a.x += re;
    a.y += im;
    amps[q] = a;
}

__global__ void k_extract(const float2 *__restrict__ root, const int32_t *__restrict__ E,
                          const int32_t *__restrict__ uniq, int64_t k, int64_t sigma, int32_t n_out, int r,
                          double2 *__restrict__ out) {
    const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= (k << r)) return;
    const int64_t p = q >> r, x = q & ((int64_t(1) << r) - 1);
    const int64_t idx = sigma * n_out + uniq[p];
    const float2 v = root[(idx << r) + root_entry(x, r)];
    out[q] = make_double2(ldexp(double(v.x), E[idx]), ldexp(double(v.y), E[idx]));
}

// Block sum of NV doubles per thread in a fixed order: lanes by xor steps,
// then the warps in turn.  Thread v < NV returns sum v.
template <int NV, int THREADS>
__device__ __forceinline__ double block_sums(double (&a)[NV], double (*part)[NV]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a[v] += __shfl_xor_sync(0xffffffffu, a[v], o);
        if (lane == 0) part[warp][v] = a[v];
    }
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < NV)
        for (int w = 0; w < THREADS / 32; ++w) s += part[w][threadIdx.x];
    return s;
}

// Sum over the blocks of a cluster (the whole grid), in rank order, by rank
// 0's first NV threads through distributed shared memory.  `mine` is this
// block's sums (thread v: sum v); returns the total there.
template <int NV>
__device__ __forceinline__ double cluster_sums(double mine, double *slot) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    if (threadIdx.x < NV) slot[threadIdx.x] = mine;
    cl.sync();
    double s = 0.0;
    if (cl.block_rank() == 0 && threadIdx.x < NV)
        for (unsigned r = 0; r < cl.num_blocks(); ++r) s += *cl.map_shared_rank(slot + threadIdx.x, r);
    cl.sync();  // the blocks' shared memory is read until here
    return s;
}

// FP64 sums over the amplitudes run on one cluster of RED_CLUSTER blocks:
// the chip's FP64 units, two lanes per SM, bound them (48 MB of amplitudes
// take 7 us of HBM; the sums below 5 to 50 FP64 operations each), so the
// more SMs the better, and a cluster adds its blocks' sums in a fixed order
// without scratch memory.
constexpr int RED_CLUSTER = 16, RED_THREADS = 512;

__global__ void __launch_bounds__(RED_THREADS) k_xeb(const double2 *__restrict__ amps, int64_t k, double scale,
                                                     double *__restrict__ out) {
    __shared__ double part[RED_THREADS / 32][1];
    __shared__ double slot[1];
    double acc[1] = {0.0};
    for (int64_t p = int64_t(blockIdx.x) * RED_THREADS + threadIdx.x; p < k; p += int64_t(gridDim.x) * RED_THREADS) {
        const double2 a = amps[p];
        acc[0] += a.x * a.x + a.y * a.y;
    }
    const double s = cluster_sums<1>(block_sums<1, RED_THREADS>(acc, part), slot);
    if (blockIdx.x == 0 && threadIdx.x == 0) out[0] = scale * s - 1.0;
}

// x = N |a|^2 in FP64 with explicit round-to-nearest operations (no
// contraction into an FMA), so that a host computing re*re + im*im, then
// times N, gets the same bits
__device__ __forceinline__ double pt_x(double2 a, double n_states) {
    return __dmul_rn(n_states, __dadd_rn(__dmul_rn(a.x, a.x), __dmul_rn(a.y, a.y)));
}

// Sums over the k amplitudes, for the mixture density
// p(x) = e^-x (1 + F (x - 1)) of x = N |amp|^2 (fidelity F; Eq. fxeb):
// out[0] = sum g, out[1] = sum g^2 with g = (x - 1) / (1 + F (x - 1)) (the
// log-likelihood's first derivative and minus its second), out[2] = sum
// log(1 + F (x - 1)), out[3] = sum x, out[4] = sum x^2.  Fixed order.
// Bound by the FP64 units: about 17 operations per amplitude, half of them
// the division, and a logarithm for every four amplitudes: log of the
// product of four d, each of them at least 1 - F > 0 (their separate
// logarithms where the product leaves the range of a double).  At F = 0 g is
// x - 1 and the logarithm 0.
//   CLUSTER: the grid is one cluster, out holds the sums;
//   else: any grid, block b writes its sums to out[5 b .. 5 b + 4], which
//   k_pt_final adds up (every SM).
// The fit of 3 M amplitudes with XEB and histogram: 1.10 ms (a pass 0.10 ms at
// F = 0, 0.12 otherwise, 0.19 with the logarithms); with one block of 1024
// threads and a logarithm each 205.7 ms.
template <bool CLUSTER>
__global__ void __launch_bounds__(RED_THREADS) k_pt_moments(const double2 *__restrict__ amps, int64_t k,
                                                            double n_states, double fid, int want_log,
                                                            double *__restrict__ out) {
    __shared__ double part[RED_THREADS / 32][5];
    __shared__ double slot[5];
    double a[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const int64_t stride = int64_t(gridDim.x) * RED_THREADS;
    auto add = [&](int64_t p) -> double {  // the sums but the logarithm's; returns d
        const double x = pt_x(amps[p], n_states);
        const double x1 = x - 1.0;
        const double d = 1.0 + fid * x1;
        const double g = fid == 0.0 ? x1 * d : x1 / d;  // (d = 1 there, NaN for an infinite x)
        a[0] += g;
        a[1] += g * g;
        a[3] += x;
        a[4] += x * x;
        if (fid == 0.0) a[2] += d - 1.0;
        return d;
    };
    int64_t p = int64_t(blockIdx.x) * RED_THREADS + threadIdx.x;
    for (; p + 3 * stride < k; p += 4 * stride) {
        double d[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) d[j] = add(p + j * stride);
        if (want_log && fid != 0.0) {
            const double q = (d[0] * d[1]) * (d[2] * d[3]);
            if (q > 1e-290 && q < 1e290) a[2] += log(q);
            else
                for (int j = 0; j < 4; ++j) a[2] += log(d[j]);
        }
    }
    for (; p < k; p += stride) {
        const double d = add(p);
        if (want_log && fid != 0.0) a[2] += log(d);
    }
    if (!want_log) a[2] = 0.0;
    const double s = block_sums<5, RED_THREADS>(a, part);
    if (CLUSTER) {
        const double t = cluster_sums<5>(s, slot);
        if (blockIdx.x == 0 && threadIdx.x < 5) out[threadIdx.x] = t;
    } else if (threadIdx.x < 5) {
        out[5 * int64_t(blockIdx.x) + threadIdx.x] = s;
    }
}

// out[v] = the sum of part[5 b + v] over the blocks b, warp v: lanes take
// every 32nd block, then xor steps (a fixed order)
__global__ void __launch_bounds__(160) k_pt_final(const double *__restrict__ part, int blocks,
                                                  double *__restrict__ out) {
    const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
    double s = 0.0;
    for (int b = lane; b < blocks; b += 32) s += part[5 * b + v];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[v] = s;
}

// counts[j] += #{b : j width <= x_b < (j + 1) width}, j < nbins, with
// width = x_max / nbins; counts[nbins] gathers x_b >= x_max.  The bin is
// floor(x / width) in FP64 (correctly rounded division), integer atomics.
__global__ void k_pt_hist(const double2 *__restrict__ amps, int64_t k, double n_states, double x_max, int nbins,
                          unsigned long long *__restrict__ counts) {
    extern __shared__ unsigned int h[];  // nbins + 1 block-local counts
    for (int j = threadIdx.x; j <= nbins; j += blockDim.x) h[j] = 0u;
    __syncthreads();
    const double width = __ddiv_rn(x_max, double(nbins));
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < k; p += int64_t(gridDim.x) * blockDim.x) {
        const double q = floor(__ddiv_rn(pt_x(amps[p], n_states), width));
        const int j = q < double(nbins) ? int(q) : nbins;
        atomicAdd(&h[j], 1u);
    }
    __syncthreads();
    for (int j = threadIdx.x; j <= nbins; j += blockDim.x)
        if (h[j]) atomicAdd(&counts[j], (unsigned long long)h[j]);
}

// Row p's batch a[p 2^r .. p 2^r + 2^r): with u = uniform[p] in [0, 1), the
// smallest x whose running sum of |a_x|^2 exceeds u times the batch total
// (2^r - 1 if none does); FP64, correctly rounded operations in x order.
//
// The running sum is a chain of dependent additions by definition, one row
// per lane (a warp instruction on the FP64 units costs the same for one lane
// as for 32).  A block takes 32 rows: four warps read the amplitudes in
// tiles of 32 rows x SAMP_T completions, coalesced, and leave |a|^2 in shared
// memory one tile ahead of warp 0, which adds up its row per lane.  It keeps
// the sum after each of at most SAMP_SEG segments; sums never decrease, so
// the first segment whose sum exceeds the threshold holds the pick, and only
// that segment is read again (8192 rows x 1024: 134 MB, 20 us of HBM, 33 M
// FP64 operations; one thread per row reading its own row twice took 632 us).
constexpr int SAMP_T = 32, SAMP_SEG = 64, SAMP_THREADS = 160;

__global__ void __launch_bounds__(SAMP_THREADS) k_sample(const double2 *__restrict__ amps, int64_t k, int r,
                                                         const double *__restrict__ uniform,
                                                         int64_t *__restrict__ picks) {
    __shared__ double s_p[2][32][SAMP_T + 1];
    __shared__ double s_ck[SAMP_SEG][32];  // running sum after each segment
    __shared__ int s_x0[32];               // first completion of the row's segment
    const int tid = threadIdx.x, lane = tid & 31;
    const bool adder = tid < 32;
    const int64_t row0 = int64_t(blockIdx.x) * 32;
    const int n = 1 << r;
    const int tb = r < 5 ? r : 5, T = 1 << tb;            // completions per tile
    const int seg = n / SAMP_SEG > T ? n / SAMP_SEG : T;  // completions per segment
    constexpr int PER = 32 * SAMP_T / (SAMP_THREADS - 32);  // entries per loading thread
    // One pass over `tiles` tiles of every row, the first at completion
    // x0(row); the adder warp calls add(p, completion within the pass) in order.
    auto pass = [&](int tiles, auto x0, auto add) {
        double2 v[PER];
        auto load = [&](int t) {
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                const int e = (tid - 32) + j * (SAMP_THREADS - 32);
                const int row = e >> tb, x = e & (T - 1);
                v[j] = make_double2(0.0, 0.0);
                if (row < 32 && row0 + row < k) v[j] = amps[((row0 + row) << r) + x0(row) + t * T + x];
            }
        };
        if (!adder) load(0);
        for (int t = 0; t < tiles; ++t) {
            if (!adder) {
#pragma unroll
                for (int j = 0; j < PER; ++j) {
                    const int e = (tid - 32) + j * (SAMP_THREADS - 32);
                    if (e < (32 << tb))
                        s_p[t & 1][e >> tb][e & (T - 1)] = __dadd_rn(__dmul_rn(v[j].x, v[j].x), __dmul_rn(v[j].y, v[j].y));
                }
                if (t + 1 < tiles) load(t + 1);
            }
            __syncthreads();  // tile t is in place; its buffer's tile t - 2 has been added up
            if (adder)
                for (int x = 0; x < T; ++x) add(s_p[t & 1][lane][x], t * T + x);
        }
        __syncthreads();
    };
    double c = 0.0;
    pass(n / T, [](int) { return 0; }, [&](double p, int x) {
        c = __dadd_rn(c, p);
        if (((x + 1) & (seg - 1)) == 0) s_ck[x / seg][lane] = c;
    });
    double thr = 0.0, c1 = 0.0;
    int x0 = 0, pick = n - 1;
    if (adder) {
        thr = __dmul_rn(row0 + lane < k ? uniform[row0 + lane] : 0.0, c);
        int j = 0;
        while (j + 1 < n / seg && !(s_ck[j][lane] > thr)) ++j;  // the last segment if none exceeds it
        x0 = j * seg;
        c1 = j > 0 ? s_ck[j - 1][lane] : 0.0;
        s_x0[lane] = x0;
    }
    __syncthreads();
    bool found = false;
    pass(seg / T, [&](int row) { return s_x0[row]; }, [&](double p, int x) {
        c1 = __dadd_rn(c1, p);
        if (!found && c1 > thr) {
            pick = x0 + x;
            found = true;
        }
    });
    if (adder && row0 + lane < k) picks[row0 + lane] = pick;
}

// FP32 fused multiply-add throughput probe: each thread runs 8 independent
// FMA chains for `iters` rounds (16 flops per round); the result is stored
// only under a condition the values never meet, so the work is kept.
__global__ void __launch_bounds__(256) k_fma_probe(int64_t iters, float seed, float *out) {
    float a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) a[j] = seed + float(threadIdx.x + j);
    const float b = 0.999999f, c = 1e-6f;
#pragma unroll 4
    for (int64_t i = 0; i < iters; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) a[j] = fmaf(a[j], b, c);
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) s += a[j];
    if (s == -1.f) out[blockIdx.x] = s;
}

}  // namespace

cudaError_t launch_fill(const FillJobD *jobs, int64_t njobs, const LeafHighD *highs, int64_t batch, float2 *ws,
                        cudaStream_t s) {
    if (njobs == 0) return cudaSuccess;
    const int64_t threads = njobs * 32;
    const int64_t blocks = (threads + 255) / 256;
    k_fill<<<dim3((unsigned)blocks), 256, 0, s>>>(jobs, njobs, highs, batch, ws);
    return cudaGetLastError();
}

// Rows of 32 and more go to k_step_narrow, the shorter ones stay in a few
// lanes' registers.
constexpr int NARROW_MIN_KB = 5;

// Lanes per row of the row kernel: as few as keep a lane's share of the
// row's K * N products within 64 (fewer cross-lane sums per output), at
// least K / 32 (a lane holds at most 32 complex A values) and at most 8
// (and K / 2: a lane loads 16 bytes at a time).
static int row_lanes(int kb, int nb) {
    const int K = 1 << kb;
    int L = (K << nb) >> 6;
    L = L < 1 ? 1 : (L > 8 ? 8 : L);
    if (L < K / 32) L = K / 32;
    if (K >= 2 && L > K / 2) L = K / 2;
    return L;
}

cudaError_t launch_step_narrow(const StepDesc &d, cudaStream_t s) {
    auto go = [&](auto kernel, int rows, int threads, size_t smem) -> cudaError_t {
        const int64_t mtiles = (int64_t(1) << d.mb) / rows;
        const int64_t nblk = d.n_ctab * mtiles;
        if (nblk <= 0) return cudaSuccess;
        if (nblk > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        kernel<<<dim3((unsigned)nblk), threads, smem, s>>>(d, (int)mtiles);
        return cudaGetLastError();
    };
    using W = NarrowTile<1, 4, 4>;
    using H = NarrowTile<2, 2, 2>;
    return (d.nInst << d.nb) <= 8 * d.n_groups ? go(k_step_narrow<2, 2, 2, 6>, H::ROWS, H::THREADS, H::SMEM)
                                               : go(k_step_narrow<1, 4, 4, 6>, W::ROWS, W::THREADS, W::SMEM);
}

bool step_narrow_takes(const StepDesc &d, bool fp32) {
    // grouped GEMMs with few columns per A instance: a tile of 64 columns is
    // mostly padding on the FMA kernel, and on the tensor cores, where B does
    // not stay resident, the loads of A and B chunk by chunk set the pace
    // (2^12 x 2^9 x 4 with 1024 A instances, 17 GB: 7.40 ms; 3.37 here).  With
    // fewer than two blocks an SM a long K would run on a few SMs
    return d.kb >= NARROW_MIN_KB && d.mb >= 7 && d.mb <= 40 && (d.nInst << d.nb) <= (fp32 ? 16 : 8) * d.n_groups &&
           (d.n_ctab << (d.mb - 7)) >= 304;
}

bool step_row_narrow(const StepDesc &d) { return d.kb >= NARROW_MIN_KB && d.mb >= 7; }

cudaError_t launch_step_row(const StepDesc &d, cudaStream_t s) {
    if (d.kb + d.nb > 8 || d.nb > 4 || d.mb > 40) return cudaErrorInvalidValue;
    if (step_row_narrow(d)) return launch_step_narrow(d, s);
    const int K = 1 << d.kb;
    const int L = row_lanes(d.kb, d.nb);
    const int R = 32 / L;
    const int KL = K / L;
    if ((d.nb == 4 && KL > 4) || (d.nb == 3 && KL > 8) || (d.nb == 2 && KL > 16) || KL > 32)
        return cudaErrorInvalidValue;  // no instance of the kernel for this split
    const int64_t M = int64_t(1) << d.mb;
    int64_t blocks, mblocks = 1;
    int rows_per_block;
    if (M >= 8 * R) {  // blocks inside one group: up to 16 (schedule 1: 4) passes of 8 warps x R rows
        int64_t passes = M / (8 * R);
        const int64_t cap = d.sched == 0 ? 16 : 4;
        passes = passes > cap ? cap : passes;
        rows_per_block = int(8 * R * passes);
        mblocks = M / rows_per_block;
        blocks = d.n_groups * mblocks;
    } else {  // small instances: 4 passes over consecutive (group, row) / schedule 1: (instance, row) pairs
        rows_per_block = 8 * R * 4;
        blocks = (((d.sched == 1 ? d.nInst : d.n_groups) << d.mb) + rows_per_block - 1) / rows_per_block;
    }
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const dim3 g((unsigned)blocks);
#define TN_ROW(NB_, KL_) k_step_row<NB_, KL_><<<g, ROW_THREADS, 0, s>>>(d, rows_per_block, mblocks)
    // KL = K / L for K * N <= 256: NB 0-1 up to 32, NB 2 up to 16, NB 3 up
    // to 8, NB 4 up to 4 (row_lanes keeps 2 KL + 2 N <= 72 registers)
#define TN_ROW_KL(NB_)                                         \
    switch (KL) {                                              \
        case 1: TN_ROW(NB_, 1); break;                         \
        case 2: TN_ROW(NB_, 2); break;                         \
        case 4: TN_ROW(NB_, 4); break;                         \
        case 8: TN_ROW(NB_, (NB_ <= 3 ? 8 : 4)); break;        \
        case 16: TN_ROW(NB_, (NB_ <= 2 ? 16 : 4)); break;      \
        default: TN_ROW(NB_, (NB_ <= 1 ? 32 : 4)); break;      \
    }
    switch (d.nb) {
        case 0: TN_ROW_KL(0); break;
        case 1: TN_ROW_KL(1); break;
        case 2: TN_ROW_KL(2); break;
        case 3: TN_ROW_KL(3); break;
        default: TN_ROW_KL(4); break;
    }
#undef TN_ROW_KL
#undef TN_ROW
    return cudaGetLastError();
}

cudaError_t launch_step_gemm_simt(const StepDesc &d, cudaStream_t s) {
    const int64_t M = int64_t(1) << d.mb;
    const int64_t N = int64_t(1) << d.nb;
    const int64_t ctiles = (int64_t(d.max_group) * N + GBN - 1) / GBN;
    const int64_t mtiles = (M + GBM - 1) / GBM;
    const int64_t blocks = d.n_groups * ctiles * mtiles;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL || ctiles > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    static_assert(SBM == GBM && SBN == GBN, "both SIMT GEMMs tile alike");
    if (d.kb >= 1) {  // K >= 2: 16-byte pieces of A rows and B columns
        k_step_gemm_simt2<<<dim3((unsigned)blocks), 128, SIMT2_SMEM, s>>>(d, (int)ctiles, (int)mtiles);
    } else {
        k_step_gemm_simt<<<dim3((unsigned)blocks), 256, 0, s>>>(d, (int)ctiles, (int)mtiles);
    }
    return cudaGetLastError();
}

// Rows side by side of a block (log2) and rows of a thread.
static int outer_rlog(const StepDesc &d) { return d.mb < 8 ? d.mb : 8; }
static int outer_rx(const StepDesc &d) { return d.mb >= 9 && d.kb <= 4 ? 2 : 1; }

bool step_outer_takes(const StepDesc &d) {
    if (d.kb > 5 || d.nb < 5 || d.mb < 5 || d.mb > 40) return false;
    if (d.kb <= 2) return true;
    // A block walks 64 columns whatever K is: with few blocks the GEMM tiles,
    // which split them, are faster (K = 16: 8 blocks 24.4 against 16.3 us, 32
    // 25 and 20, 64 25 and 27; K = 8: 37 blocks 19 and 18, 64 14 and 18; K =
    // 32: 16 blocks 24 and 20, 32 17 and 21)
    const int64_t blocks = d.n_ctab * ((int64_t(1) << d.mb) / (outer_rx(d) << outer_rlog(d)));
    return blocks >= (d.kb == 5 ? 32 : 48);
}

cudaError_t launch_step_outer(const StepDesc &d, cudaStream_t s) {
    if (!step_outer_takes(d)) return cudaErrorInvalidValue;
    const int rlog = outer_rlog(d), rx = outer_rx(d);
    // up to four passes of rows for one B tile, while that leaves eight blocks an SM
    int passes = 1;
    const int64_t tiles = (int64_t(1) << d.mb) / (rx << rlog);
    while (passes < 4 && passes < tiles && d.n_ctab * (tiles / (2 * passes)) >= 1216) passes *= 2;
    const int64_t mtiles = tiles / passes, blocks = d.n_ctab * mtiles;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const dim3 g((unsigned)blocks);
#define TN_OUTER(KB_)                                                                   \
    do {                                                                                \
        if (rx == 2) k_step_outer<KB_, 2><<<g, 256, 0, s>>>(d, rlog, passes, (int)mtiles); \
        else k_step_outer<KB_, 1><<<g, 256, 0, s>>>(d, rlog, passes, (int)mtiles);      \
    } while (0)
    switch (d.kb) {
        case 0: TN_OUTER(0); break;
        case 1: TN_OUTER(1); break;
        case 2: TN_OUTER(2); break;
        case 3: TN_OUTER(3); break;
        case 4: TN_OUTER(4); break;
        default: k_step_outer<5, 1><<<g, 256, 0, s>>>(d, rlog, passes, (int)mtiles); break;
    }
#undef TN_OUTER
    return cudaGetLastError();
}

bool step_skinny_takes(const StepDesc &d) { return d.kb >= 6 && d.nb <= 3 && d.mb + d.nb <= 5; }

cudaError_t launch_step_skinny(const StepDesc &d, cudaStream_t s) {
    if (!step_skinny_takes(d)) return cudaErrorInvalidValue;
    const int rmb = d.mb < 3 - d.nb ? d.mb : 3 - d.nb;  // RM N <= 8
    const int64_t units = d.nInst << (d.mb - rmb);
    if (units <= 0) return cudaSuccess;
    // a block per unit where its 256 lanes have several pieces each, or
    // where one warp per unit would leave most of the chip idle
    const bool wide = d.kb >= 12 || (d.kb >= 9 && units < 4864);
    const int64_t blocks = wide ? units : (units + 7) / 8;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    const dim3 g((unsigned)blocks);
#define TN_SKINNY(RM_, N_)                                                 \
    do {                                                                   \
        if (wide) k_step_skinny<RM_, N_, 8><<<g, 256, 0, s>>>(d, units);   \
        else k_step_skinny<RM_, N_, 1><<<g, 256, 0, s>>>(d, units);        \
    } while (0)
    switch (4 * d.nb + rmb) {
        case 0: TN_SKINNY(1, 1); break;
        case 1: TN_SKINNY(2, 1); break;
        case 2: TN_SKINNY(4, 1); break;
        case 3: TN_SKINNY(8, 1); break;
        case 4: TN_SKINNY(1, 2); break;
        case 5: TN_SKINNY(2, 2); break;
        case 6: TN_SKINNY(4, 2); break;
        case 8: TN_SKINNY(1, 4); break;
        case 9: TN_SKINNY(2, 4); break;
        default: TN_SKINNY(1, 8); break;
    }
#undef TN_SKINNY
    return cudaGetLastError();
}

cudaError_t init_simt_kernels() {
    const cudaError_t e =
        cudaFuncSetAttribute(k_step_narrow<1, 4, 4, 6>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(NarrowTile<1, 4, 4>::SMEM));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_step_gemm_simt2, cudaFuncAttributeMaxDynamicSharedMemorySize, int(SIMT2_SMEM));
}

cudaError_t launch_accumulate(const float2 *root, const int32_t *E, const int32_t *uniq, int64_t k,
                              int64_t n_sig, int32_t n_out, int r, double *amps, cudaStream_t s) {
    if (k == 0) return cudaSuccess;
    if (r < 0 || r > 30) return cudaErrorInvalidValue;
    const int64_t blocks = ((k << r) + 255) / 256;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    k_accumulate<<<dim3((unsigned)blocks), 256, 0, s>>>(root, E, uniq, k, n_sig, n_out, r,
                                                        reinterpret_cast<double2 *>(amps));
    return cudaGetLastError();
}

cudaError_t launch_extract(const float2 *root, const int32_t *E, const int32_t *uniq, int64_t k, int64_t sigma,
                           int32_t n_out, int r, double *out, cudaStream_t s) {
    if (k == 0) return cudaSuccess;
    if (r < 0 || r > 30) return cudaErrorInvalidValue;
    const int64_t blocks = ((k << r) + 255) / 256;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    k_extract<<<dim3((unsigned)blocks), 256, 0, s>>>(root, E, uniq, k, sigma, n_out, r,
                                                     reinterpret_cast<double2 *>(out));
    return cudaGetLastError();
}

// one cluster as the whole grid, no more blocks than have work (a power of
// two; a few thousand amplitudes stay on one SM)
template <class... P, class... A>
static cudaError_t launch_cluster(void (*fn)(P...), int64_t k, int64_t per_block, cudaStream_t s, A... args) {
    unsigned blocks = 1;
    while (blocks < unsigned(RED_CLUSTER) && blocks * per_block < k) blocks <<= 1;
    cudaError_t e = cudaSuccess;
    if (blocks > 8)
        e = cudaFuncSetAttribute(reinterpret_cast<const void *>(fn), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(RED_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = blocks > 1 ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, fn, args...);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_xeb(const double *amps, int64_t k, double scale, double *out, cudaStream_t s) {
    return launch_cluster(k_xeb, k, RED_THREADS, s, reinterpret_cast<const double2 *>(amps), k, scale, out);
}

// Batches of at most 32 completions: a row per thread, its |a|^2 in registers,
// so neither a tile nor a second read (8 completions: 256 rows 8.2 us in tiles,
// 4.1 here; 65536 rows of 16: 39 and 16.5, of 32: 49 and 28.9).
template <int R>
__global__ void __launch_bounds__(128) k_sample_rows(const double2 *__restrict__ amps, int64_t k,
                                                     const double *__restrict__ uniform, int64_t *__restrict__ picks) {
    constexpr int N = 1 << R, H = N < 16 ? N : 16;  // loads in flight
    const int64_t p = int64_t(blockIdx.x) * 128 + threadIdx.x;
    if (p >= k) return;
    const double u = uniform[p];
    double w[N], tot = 0.0;
#pragma unroll
    for (int h = 0; h < N; h += H) {
        double2 v[H];
#pragma unroll
        for (int x = 0; x < H; ++x) v[x] = amps[(p << R) + h + x];
#pragma unroll
        for (int x = 0; x < H; ++x) {
            w[h + x] = __dadd_rn(__dmul_rn(v[x].x, v[x].x), __dmul_rn(v[x].y, v[x].y));
            tot = __dadd_rn(tot, w[h + x]);
        }
    }
    const double thr = __dmul_rn(u, tot);
    double c = 0.0;
    int pick = N - 1;
    bool open = true;
#pragma unroll
    for (int x = 0; x < N; ++x) {
        c = __dadd_rn(c, w[x]);
        if (open && c > thr) {
            pick = x;
            open = false;
        }
    }
    picks[p] = pick;
}

cudaError_t launch_sample(const double *amps, int64_t k, int r, const double *uniform, int64_t *picks,
                          cudaStream_t s) {
    if (k == 0) return cudaSuccess;
    if (r <= 5) {
        const int64_t blocks = (k + 127) / 128;
        if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
        const double2 *a = reinterpret_cast<const double2 *>(amps);
        const dim3 g((unsigned)blocks);
        switch (r) {
            case 0: k_sample_rows<0><<<g, 128, 0, s>>>(a, k, uniform, picks); break;
            case 1: k_sample_rows<1><<<g, 128, 0, s>>>(a, k, uniform, picks); break;
            case 2: k_sample_rows<2><<<g, 128, 0, s>>>(a, k, uniform, picks); break;
            case 3: k_sample_rows<3><<<g, 128, 0, s>>>(a, k, uniform, picks); break;
            case 4: k_sample_rows<4><<<g, 128, 0, s>>>(a, k, uniform, picks); break;
            default: k_sample_rows<5><<<g, 128, 0, s>>>(a, k, uniform, picks); break;
        }
        return cudaGetLastError();
    }
    const int64_t blocks = (k + 31) / 32;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    k_sample<<<dim3((unsigned)blocks), SAMP_THREADS, 0, s>>>(reinterpret_cast<const double2 *>(amps), k, r, uniform,
                                                             picks);
    return cudaGetLastError();
}

// An SM's two FP64 lanes take 1 us for about 50 amplitudes' sums, so a few
// amplitudes already spread over the cluster.
constexpr int64_t PT_PER_SM = 64;

cudaError_t launch_pt_moments(const double *amps, int64_t k, double n_states, double fid, double *out,
                              cudaStream_t s) {
    return launch_cluster(k_pt_moments<true>, k, PT_PER_SM, s, reinterpret_cast<const double2 *>(amps), k, n_states,
                          fid, 1, out);
}

// Blocks of the scratch form: an amplitude a thread at least, at most
// PT_BLOCKS (two resident blocks on each of 152 SMs).
constexpr int PT_BLOCKS = 304;
static int pt_blocks(int64_t k) {
    const int64_t b = (k + RED_THREADS - 1) / RED_THREADS;
    return int(b < 1 ? 1 : (b > PT_BLOCKS ? PT_BLOCKS : b));
}

size_t pt_moments_scratch_bytes(int64_t k) { return size_t(pt_blocks(k)) * 5 * sizeof(double); }

cudaError_t launch_pt_moments_scratch(const double *amps, int64_t k, double n_states, double fid, bool want_log,
                                      double *out, double *scratch, cudaStream_t s) {
    const int blocks = pt_blocks(k);
    if (blocks <= RED_CLUSTER)  // one launch instead of two (a fit of 1000 amplitudes: 366 -> 310 us)
        return launch_cluster(k_pt_moments<true>, k, PT_PER_SM, s, reinterpret_cast<const double2 *>(amps), k,
                              n_states, fid, want_log ? 1 : 0, out);
    k_pt_moments<false><<<blocks, RED_THREADS, 0, s>>>(reinterpret_cast<const double2 *>(amps), k, n_states, fid,
                                                       want_log ? 1 : 0, scratch);
    k_pt_final<<<1, 160, 0, s>>>(scratch, blocks, out);
    return cudaGetLastError();
}

cudaError_t launch_pt_hist(const double *amps, int64_t k, double n_states, double x_max, int nbins,
                           unsigned long long *counts, cudaStream_t s) {
    const int64_t want = (k + 255) / 256;
    const int blocks = int(want < 1024 ? (want > 0 ? want : 1) : 1024);
    k_pt_hist<<<blocks, 256, size_t(nbins + 1) * sizeof(unsigned int), s>>>(reinterpret_cast<const double2 *>(amps),
                                                                         k, n_states, x_max, nbins, counts);
    return cudaGetLastError();
}

cudaError_t launch_fma_probe(int64_t blocks, int64_t iters, float *out, cudaStream_t s) {
    if (blocks <= 0 || blocks > 0x7fffffffLL || iters < 0) return cudaErrorInvalidValue;
    k_fma_probe<<<dim3((unsigned)blocks), 256, 0, s>>>(iters, 1.0f, out);
    return cudaGetLastError();
}

}  // namespace tnk
