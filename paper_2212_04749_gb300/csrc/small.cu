// Small steps, many to a launch.
//
// Below a few 10^5 multiply-adds a pairwise step costs what any launch
// costs: the launch itself, its wait for the previous step and four or five
// dependent loads, about 5 us, and a contraction has tens to hundreds of such
// steps (the merges of leaf tensors and the tail near the root).  Here one
// cluster of up to 16 blocks runs a list of them: the steps are sorted into
// phases on the host, a phase's steps depend on earlier phases only and run
// side by side, and a cluster barrier between phases takes the place of the
// launch.  A phase costs its barrier and one round trip to L2 (maxima,
// exponents, A and B together), about 2.5 us of ten with the launch; a warp looks up its part of the next phase and
// the instances there between its arrival at the barrier and the wait.
// 64 amplitudes of 3x4 with 8 cycles: 34.9 us with the look-up and the
// exponents' loads behind the barrier, 32.6 so; as separate launches 177.
//
// An output C[i](m, n) is one sum over k, split over 2^lanes_log2
// neighbouring lanes where a step has fewer outputs than the cluster has
// threads, in FP32 FMA; rescale and exponents as in the other step kernels.
// Operands written by an earlier phase of the same launch come from other
// SMs, so they are read past L1 (ld.global.cg).
#include <cstring>

#include "kernels.cuh"

namespace tnk {

namespace {

// The latencies of a phase count per thread, so more threads of fewer outputs
// each are better until their registers spill: 256, 512 and 1024 a block take
// 106, 102.5 and 103 us for 500 amplitudes of 4x5 with 7 cycles, 78, 70 and 72
// us for 33 of 5x5 with 6 (1024 have 64 registers each and spill).
constexpr int SM_THREADS = 512, SM_WARPS = SM_THREADS / 32;
constexpr int SM_CLUSTER = 16;

__device__ __forceinline__ void sm_cfma(float2 &acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// The instances of output `first + lane` of a step (the last one's where
// there is none): nothing that an earlier phase writes.
__device__ __forceinline__ int2 small_instances(const SmallDesc &d, int lg, int first, int lane) {
    const int o = (first + lane) >> lg;
    return __ldg(d.instab + ((o < d.outputs ? o : 0) >> d.mnb));
}

// U x 32 lanes of one step (lane groups of 2^lg lanes, one output each), U
// outputs a lane at once so that their loads are in flight together; ab0: the
// first ones' instances (small_instances).
template <int U>
__device__ __forceinline__ void small_outputs(const SmallDesc &d, int lg, int first, int lane, int2 ab0) {
    const int sub = lane & ((1 << lg) - 1);
    bool valid[U];
    int i[U], mn[U];
    int2 ab[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int o = (first + 32 * u + lane) >> lg;
        valid[u] = o < d.outputs;
        const int oc = valid[u] ? o : 0;
        i[u] = oc >> d.mnb;
        mn[u] = oc & ((1 << d.mnb) - 1);
        ab[u] = u == 0 ? ab0 : __ldg(d.instab + i[u]);
    }
    uint32_t ma[U], mb[U];
    int32_t Ea[U], Eb[U];  // loaded with the operands: at the end they would be one more round trip
    const float2 *a[U], *b[U];
    float2 acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        ma[u] = d.mxA ? __ldcg(d.mxA + ab[u].x) : 0u;
        mb[u] = d.mxB ? __ldcg(d.mxB + ab[u].y) : 0u;
        const bool first_of = mn[u] == 0 && sub == 0;
        Ea[u] = first_of ? __ldcg(d.EA + ab[u].x) : 0;
        Eb[u] = first_of ? __ldcg(d.EB + ab[u].y) : 0;
        a[u] = d.A + int64_t(ab[u].x) * d.sA + (int64_t(mn[u] >> d.nb) << d.kb);
        b[u] = d.B + int64_t(ab[u].y) * d.sB + (int64_t(mn[u] & ((1 << d.nb) - 1)) << d.kb);
        acc[u] = make_float2(0.f, 0.f);
    }
    if (d.kb == 0) {
        float2 x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = __ldcg(a[u]);
            y[u] = __ldcg(b[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) sm_cfma(acc[u], x[u], y[u]);
    } else {
        const int pieces = 1 << (d.kb - 1);
#pragma unroll(U == 1 ? 4 : 2)
        for (int q = sub; q < pieces; q += 1 << lg) {
            float4 x[U], y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                x[u] = __ldcg(reinterpret_cast<const float4 *>(a[u]) + q);
                y[u] = __ldcg(reinterpret_cast<const float4 *>(b[u]) + q);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                sm_cfma(acc[u], make_float2(x[u].x, x[u].y), make_float2(y[u].x, y[u].y));
                sm_cfma(acc[u], make_float2(x[u].z, x[u].w), make_float2(y[u].z, y[u].w));
            }
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        for (int s = 1; s < (1 << lg); s <<= 1) {  // lg is the same for the warp
            acc[u].x += __shfl_xor_sync(0xffffffffu, acc[u].x, s);
            acc[u].y += __shfl_xor_sync(0xffffffffu, acc[u].y, s);
        }
        const int ea = exp_of(ma[u]), eb = exp_of(mb[u]);
        const float sc = pow2f(-(ea + eb));
        const float2 v = make_float2(acc[u].x * sc, acc[u].y * sc);
        uint32_t mx = 0u;
        if (valid[u] && sub == 0) {
            int64_t c = int64_t(i[u]) * d.sC;
            for (int j = 0; j < d.mnb; ++j) c += int64_t((mn[u] >> j) & 1) << d.pC[j];
            d.C[c] = v;
            if (mn[u] == 0) d.EC[i[u]] = Ea[u] + ea + Eb[u] + eb;
            mx = __float_as_uint(fmaxf(fabsf(v.x), fabsf(v.y)));
        }
        if (d.mxC) {
            if (d.mnb + lg >= 5) {  // one instance for the 32 lanes
                mx = __reduce_max_sync(0xffffffffu, mx);
                if (lane == 0 && mx) atomicMax(d.mxC + i[u], mx);
            } else if (mx) {
                atomicMax(d.mxC + i[u], mx);
            }
        }
    }
}

__global__ void __launch_bounds__(SM_THREADS) k_small_steps(const __grid_constant__ SmallArgs p) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    SmallDesc *sd = reinterpret_cast<SmallDesc *>(sm_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int PIECES = int(sizeof(SmallDesc) / 16);
    for (int e = tid; e < p.n_steps * PIECES; e += SM_THREADS) {
        const int s = e / PIECES, q = e - s * PIECES;
        reinterpret_cast<uint4 *>(sd + s)[q] = __ldg(reinterpret_cast<const uint4 *>(p.descs + p.step[s]) + q);
    }
    __syncthreads();
    const int nw = int(gridDim.x) * SM_WARPS, gw = int(blockIdx.x) + warp * int(gridDim.x);
    int s0 = 0, s1 = p.phase_end[0], s = 0, local = 0;
    // the step and place of the phase's warp w (s: from the phase's first step on)
    auto locate = [&](int w) {
        while (w >= p.wend[s]) ++s;
        local = w - (s > s0 ? p.wend[s - 1] : 0);
    };
    auto instances = [&] {
        return small_instances(sd[s], p.lanes_log2[s], local * (p.four[s] ? 128 : 32), lane);
    };
    int2 ab = make_int2(0, 0);
    bool mine = gw < p.wend[s1 - 1];
    if (mine) {
        locate(gw);
        ab = instances();
    }
    for (int ph = 0;;) {
        for (int w = gw; mine;) {
            if (p.four[s]) small_outputs<4>(sd[s], p.lanes_log2[s], local * 128, lane, ab);
            else small_outputs<1>(sd[s], p.lanes_log2[s], local * 32, lane, ab);
            w += nw;
            mine = w < p.wend[s1 - 1];
            if (mine) {
                locate(w);
                ab = instances();
            }
        }
        if (++ph == p.n_phases) break;
        // release: this phase's outputs, maxima and exponents; meanwhile the
        // next phase's place and instances, which depend on none of them
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        s = s0 = s1;
        s1 = p.phase_end[ph];
        mine = gw < p.wend[s1 - 1];
        if (mine) {
            locate(gw);
            ab = instances();
        }
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}

// One step of few multiply-adds, too many for the cluster: an output per group
// of 2^lg lanes over the whole chip, rows of A in neighbouring lanes (they are
// neighbours in C where the layout allows).  Operands come through L1: 16
// bytes a multiply-add.  Latency-bound: the tiled kernels put such a step on
// a few SMs and walk K serially there (2^11 x 32 x 32 in FP32 16.3 us, 8.2
// here; 2^15 x 8 x 8 24.8 and 10.0 on the row kernel; 33 instances of 2^4 x 64
// x 8 26.1 and 6.0).  (d.nb: the row bits, which come first in pC.)
constexpr int FEW_THREADS = 256;

__global__ void __launch_bounds__(FEW_THREADS) k_step_few(const __grid_constant__ SmallDesc d, int lg) {
    __shared__ uint32_t s_mx;
    const int t = int(blockIdx.x) * FEW_THREADS + int(threadIdx.x), sub = t & ((1 << lg) - 1), o = t >> lg;
    const bool valid = o < d.outputs, one = d.mnb + lg >= 8;  // one: a block's outputs belong to one instance
    const int oc = valid ? o : 0, i = oc >> d.mnb, mn = oc & ((1 << d.mnb) - 1);
    if (threadIdx.x == 0) s_mx = 0u;
    if (d.mxC && one) __syncthreads();
    const int2 ab = __ldg(d.instab + i);
    const uint32_t ma = d.mxA ? __ldg(d.mxA + ab.x) : 0u, mb = d.mxB ? __ldg(d.mxB + ab.y) : 0u;
    const float2 *a = d.A + int64_t(ab.x) * d.sA + (int64_t(mn & ((1 << d.nb) - 1)) << d.kb);
    const float2 *b = d.B + int64_t(ab.y) * d.sB + (int64_t(mn >> d.nb) << d.kb);
    int64_t c = int64_t(i) * d.sC;
    for (int j = 0; j < d.mnb; ++j) c += int64_t((mn >> j) & 1) << d.pC[j];
    float2 acc = make_float2(0.f, 0.f);
    if (d.kb == 0) {
        sm_cfma(acc, __ldg(a), __ldg(b));
    } else {
        const int pieces = 1 << (d.kb - 1);
#pragma unroll 4
        for (int q = sub; q < pieces; q += 1 << lg) {
            const float4 x = __ldg(reinterpret_cast<const float4 *>(a) + q);
            const float4 y = __ldg(reinterpret_cast<const float4 *>(b) + q);
            sm_cfma(acc, make_float2(x.x, x.y), make_float2(y.x, y.y));
            sm_cfma(acc, make_float2(x.z, x.w), make_float2(y.z, y.w));
        }
    }
    for (int s = 1; s < (1 << lg); s <<= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, s);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, s);
    }
    const int ea = exp_of(ma), eb = exp_of(mb);
    const float sc = pow2f(-(ea + eb));
    const float2 v = make_float2(acc.x * sc, acc.y * sc);
    uint32_t mx = 0u;
    if (valid && sub == 0) {
        d.C[c] = v;
        if (mn == 0) d.EC[i] = __ldg(d.EA + ab.x) + ea + __ldg(d.EB + ab.y) + eb;
        mx = __float_as_uint(fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    if (!d.mxC) return;
    if (one) {
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((threadIdx.x & 31) == 0 && mx) atomicMax(&s_mx, mx);
        __syncthreads();
        if (threadIdx.x == 0 && s_mx) atomicMax(d.mxC + i, s_mx);
    } else if (d.mnb + lg >= 5) {
        mx = __reduce_max_sync(0xffffffffu, mx);
        if ((threadIdx.x & 31) == 0 && mx) atomicMax(d.mxC + i, mx);
    } else if (mx) {
        atomicMax(d.mxC + i, mx);
    }
}

}  // namespace

bool step_few_takes(const StepDesc &d, bool tc, bool own) {
    // 2^23 multiply-adds (128 MB through L1, 4 us); against the tensor cores,
    // whose persistent kernel takes 14 us for any small step, 2^21: 2^14 x 16 x
    // 16 takes 16.3 us here and 14.2 there, 2^11 x 32 x 32 8.2 and 16.3.
    // Single outputs of K = 2^9 and more are the skinny kernel's: 12.1 us here
    // against 8.0 at K = 2^10
    if (d.kb > 10 || d.mb + d.nb > 20 || (d.kb >= 9 && step_skinny_takes(d))) return false;
    const int64_t out = d.nInst << (d.mb + d.nb), macs = out << d.kb, one = 1;
    if (out > (one << 20) || macs > (one << (tc ? 21 : 23))) return false;
    // 2^18 outputs and more: K <= 8, 2^22 multiply-adds where the row kernel
    // cannot take it (2^18 outputs of K = 32 in a GEMM: 26.5 us here, 20.4
    // there; 2^20 of K = 8 19.6 and 18.0)
    const bool row = d.nb <= 4 && d.kb + d.nb <= 8;
    if (out > (one << 17) && (d.kb > 3 || macs > (one << (row ? 23 : 22)))) return false;
    // Beyond this the row kernel's second schedule is often faster (2^18 x 4 x 4
    // 18.5 us here, 15.7 under configuration 0, 9.8 under 1; 2^15 x 32 x 8 24.4,
    // 24.4 and 12.1), so there only in the place of the plan's own
    // configuration: tuning tells them apart
    return own || out <= (one << 16) || (out <= (one << 18) && macs <= (one << 21));
}

cudaError_t launch_step_few(const StepDesc &d, cudaStream_t s) {
    if (!step_few_takes(d, false, true)) return cudaErrorInvalidValue;
    SmallDesc r;
    std::memset(&r, 0, sizeof(r));
    r.A = d.A;
    r.B = d.B;
    r.C = d.C + d.inst0 * d.sC;
    r.instab = d.instab + d.inst0;
    r.EA = d.EA;
    r.EB = d.EB;
    r.EC = d.EC + d.inst0;
    r.mxA = d.mxA;
    r.mxB = d.mxB;
    r.mxC = d.mxC ? d.mxC + d.inst0 : nullptr;
    r.sA = d.sA;
    r.sB = d.sB;
    r.sC = d.sC;
    r.kb = (int8_t)d.kb;
    r.nb = (int8_t)d.mb;
    r.mnb = (int8_t)(d.mb + d.nb);
    r.outputs = (int32_t)(d.nInst << (d.mb + d.nb));
    for (int j = 0; j < d.mb; ++j) r.pC[j] = d.pCm[j];
    for (int j = 0; j < d.nb; ++j) r.pC[d.mb + j] = d.pCn[j];
    if (r.outputs <= 0) return cudaSuccess;
    // lanes per output: while the chip has threads to spare and a lane two entries
    int lg = 0;
    while (lg < 5 && lg < d.kb - 1 && (int64_t(r.outputs) << (lg + 1)) <= 131072) ++lg;
    const int64_t blocks = ((int64_t(r.outputs) << lg) + FEW_THREADS - 1) / FEW_THREADS;
    k_step_few<<<dim3((unsigned)blocks), FEW_THREADS, 0, s>>>(r, lg);
    return cudaGetLastError();
}

cudaError_t init_small_kernel() {
    cudaError_t e = cudaFuncSetAttribute(k_small_steps, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(SMALL_MAX_STEPS * sizeof(SmallDesc)));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_small_steps, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t launch_small(const SmallArgs &a, cudaStream_t s) {
    if (a.n_steps < 1 || a.n_steps > SMALL_MAX_STEPS || a.n_phases < 1 || a.n_phases > SMALL_MAX_PHASES)
        return cudaErrorInvalidValue;
    // as many blocks as the widest phase has work for: a barrier over fewer
    // blocks is shorter
    unsigned blocks = 1;
    while (blocks < unsigned(SM_CLUSTER) && int(blocks) * SM_WARPS < a.max_warps) blocks <<= 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(SM_THREADS);
    cfg.dynamicSmemBytes = size_t(a.n_steps) * sizeof(SmallDesc);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_small_steps, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace tnk
