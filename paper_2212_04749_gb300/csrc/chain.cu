// Fused chain of small-operand steps (SM Sec. V.C: a tile of the big tensor
// stays in fast memory while the chain's small tensors are applied to it,
// and only the chain's last output is written back).
//
// Chain s_1 .. s_L:  C_j(m, n) = sum_k C_{j-1}(k, m) B_j(k, n), C_0 = A_1.
// Bits of A_1 that no chain step contracts pass through to C_L; some of them
// (the outside bits O) number the tiles, the others are tile bits: those the
// chain contracts or produces, and more, from the low address bits of A_1 and
// C_L, up to 2^12 entries, so that a tile is read and written in contiguous
// runs.  A block
//   1. loads an A_1 tile by 16-byte cp.async into shared memory,
//   2. applies B_1 .. B_L (staged once per block) tile to tile, ping-ponging
//      between two buffers; a thread takes rows: K neighbouring entries in
//      registers against every column of B_j (in registers too where K N <=
//      16),
//   3. scales by the operands' power-of-two factors and writes the C_L tile
//      through its address bits, 16 bytes a store.
// Tile index bits are the tile's address bits in ascending order, so the
// contracted bits of every step are the lowest bits of its input tile (the
// planner keeps every operand K-major) and row r's K inputs are entries
// K r .. K r + K - 1.  An index is the OR of a thread's part (a small table) and
// a part of the round (in the kernel's parameters): no per-entry tables.
//
// Bound: one read of A_1 and one write of C_L at HBM (L2) speed against L
// passes of 4 N fused multiply-adds and one shared-memory round trip an entry;
// six steps of K = N = 4 issue in 62 % of the cycles (FMA pipe 33 %, shared
// memory 45 %, DRAM 13 %), the rest waits at the barriers between steps.  Six such
// steps on 2^23 entries (134 MB, 20 us of HBM) take 85 us, 33-43 us each as
// separate row kernels; the kernel before, a warp per tile of at most 2^10
// with 8-byte loads through per-entry index tables, took 570 us (2^7) to 6 ms
// (2^10) for chains of this size.
//
// Rescale: B_j is multiplied by 2^-eb_j, the exponent of its largest component,
// as it is staged, C_L by 2^-ea, and its exponent is
// E_A + ea + sum_j (E_Bj + eb_j).  So the intermediates, which are not rescaled
// themselves, stay in range whatever the side operands' scale.  Power-of-two
// factors are exact.
#include "kernels.cuh"

namespace tnk {

namespace {

constexpr int CH_MAX_THREADS = 256;

__device__ __forceinline__ void ch_record_max(uint32_t *slot, uint32_t v) {
    asm volatile("red.relaxed.gpu.global.max.u32 [%0], %1;" ::"l"(slot), "r"(v) : "memory");
}

// Tile buffers are XOR-swizzled in 16-byte units (pairs of entries): bits 1-3
// of an entry index take bits 4-6 and 7-9, so that threads whose entries lie
// a power of two apart use different banks.  Linear over GF(2): the swizzle
// of an OR of disjoint parts is the XOR of the parts' swizzles.
__device__ __forceinline__ int swz(int i) { return i ^ ((((i >> 4) ^ (i >> 7)) & 7) << 1); }

__device__ __forceinline__ void cmac(float2 &acc, float2 u, float2 v) {
    acc.x = fmaf(u.x, v.x, acc.x);
    acc.x = fmaf(-u.y, v.y, acc.x);
    acc.y = fmaf(u.x, v.y, acc.y);
    acc.y = fmaf(u.y, v.x, acc.y);
}

// K entries of the row whose first (swizzled) entry is at
template <int KB>
__device__ __forceinline__ void load_row(float2 (&x)[1 << KB], const float2 *xi, int at) {
    if (KB == 0) {
        x[0] = xi[at];
    } else {
#pragma unroll
        for (int q = 0; q < (1 << KB) / 2; ++q) {  // 2 q < 16: its swizzle is itself
            const float4 v = *reinterpret_cast<const float4 *>(xi + (at ^ (2 * q)));
            x[2 * q] = make_float2(v.x, v.y);
            x[2 * q + 1] = make_float2(v.z, v.w);
        }
    }
}

// One step's view for a thread: where rows and columns go in the output tile.
struct StepView {
    const float2 *B;      // [N][K] in shared memory
    const int8_t *cpos;   // output tile bit of each n bit
    const int16_t *col;   // N <= 16: swizzled output part of each column
    const int16_t *rowhi; // swizzled output part of each round
    int kb, nb, rbits;    // rows: 2^rbits
    int rowlo;            // this thread's swizzled output part
    bool pairs;           // columns 2 e, 2 e + 1 are neighbours in the output

    __device__ __forceinline__ int column(int n) const {
        if (nb <= 4) return col[n];
        int c = 0;
        for (int q = 0; q < nb; ++q) c |= ((n >> q) & 1) << cpos[q];
        return swz(c);
    }
};

// K and N compile-time, K N <= 16: B in registers for all of the thread's
// rows; neighbouring columns are stored 16 bytes at a time.
template <int KB, int NB>
__device__ __forceinline__ void step_regs(const StepView &v, const float2 *xi, float2 *xo, int t, int TH) {
    constexpr int K = 1 << KB, N = 1 << NB;
    float2 b[N][K];
    int col[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        col[n] = v.col[n];
        if (K == 1) {
            b[n][0] = v.B[n];
        } else {
#pragma unroll
            for (int q = 0; q < K / 2; ++q) {
                const float4 x = *reinterpret_cast<const float4 *>(v.B + n * K + 2 * q);
                b[n][2 * q] = make_float2(x.x, x.y);
                b[n][2 * q + 1] = make_float2(x.z, x.w);
            }
        }
    }
    const int R = 1 << v.rbits;
#pragma unroll 2
    for (int r = t, i = 0; r < R; r += TH, ++i) {
        float2 x[K];
        load_row<KB>(x, xi, swz(r << KB));
        const int row = v.rowlo ^ v.rowhi[i];
        float2 acc[N];
#pragma unroll
        for (int n = 0; n < N; ++n) {
            acc[n] = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k) cmac(acc[n], x[k], b[n][k]);
        }
        if (NB > 0 && v.pairs) {
#pragma unroll
            for (int n = 0; n + 1 < N; n += 2)
                *reinterpret_cast<float4 *>(xo + (row ^ col[n])) =
                    make_float4(acc[n].x, acc[n].y, acc[n + 1].x, acc[n + 1].y);
        } else {
#pragma unroll
            for (int n = 0; n < N; ++n) xo[row ^ col[n]] = acc[n];
        }
    }
}

// K compile-time, any N: B as warp broadcasts; with fewer rows than threads
// the columns are dealt to the threads as well.
template <int KB>
__device__ __forceinline__ void step_cols(const StepView &v, const float2 *xi, float2 *xo, int t, int TH) {
    constexpr int K = 1 << KB;
    const int R = 1 << v.rbits, N = 1 << v.nb;
    int n0 = 0, n1 = N, r0 = t;
    if (R < TH) {
        const int per = max(1, (N * R) / TH);  // columns per thread
        r0 = t & (R - 1);
        n0 = (t >> v.rbits) * per;
        n1 = n0 < N ? n0 + per : n0;
    }
    for (int r = r0, i = 0; r < R; r += TH, ++i) {
        float2 x[K];
        load_row<KB>(x, xi, swz(r << KB));
        const int row = v.rowlo ^ v.rowhi[i];
        for (int n = n0; n < n1; ++n) {
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll
            for (int k = 0; k < K; ++k) cmac(acc, x[k], v.B[n * K + k]);
            xo[row ^ v.column(n)] = acc;
        }
    }
}

// K above 16: the row's entries from shared memory as well.
__device__ __forceinline__ void step_long(const StepView &v, const float2 *xi, float2 *xo, int t, int TH) {
    const int R = 1 << v.rbits, N = 1 << v.nb, K = 1 << v.kb;
    int n0 = 0, n1 = N, r0 = t;
    if (R < TH) {
        const int per = max(1, (N * R) / TH);
        r0 = t & (R - 1);
        n0 = (t >> v.rbits) * per;
        n1 = n0 < N ? n0 + per : n0;
    }
    for (int r = r0, i = 0; r < R; r += TH, ++i) {
        const int row = v.rowlo ^ v.rowhi[i];
        for (int n = n0; n < n1; ++n) {
            float2 acc = make_float2(0.f, 0.f);
            for (int k = 0; k < K; ++k) cmac(acc, xi[swz((r << v.kb) | k)], v.B[n * K + k]);
            xo[row ^ v.column(n)] = acc;
        }
    }
}

__global__ void __launch_bounds__(CH_MAX_THREADS, 3) k_chain(const __grid_constant__ ChainDesc d) {
    extern __shared__ __align__(16) unsigned char ch_raw[];
    __shared__ int s_boff[CH_MAXL + 1];
    __shared__ float s_sc;
    __shared__ uint32_t s_mx;
    __shared__ int32_t s_tab[CH_MAXL + 1], s_e[CH_MAXL + 1], s_E[CH_MAXL + 1];
    const int t = threadIdx.x, lane = t & 31, TH = blockDim.x;
    const int64_t inst = d.inst0 + int64_t(blockIdx.x) / d.oblocks;
    const int64_t ob = int64_t(blockIdx.x) % d.oblocks;
    const int L = d.L, tout = d.tb[L - 1];
    if (t <= L) {
        const int id = __ldg(d.tab + inst * (L + 1) + t);
        const uint32_t *mx = t == 0 ? d.mxA : d.mxB[t - 1];
        const int32_t *E = t == 0 ? d.EA : d.EB[t - 1];
        const int e = mx ? exp_of(mx[id]) : 0;
        s_tab[t] = id;
        s_e[t] = e;
        s_E[t] = E[id] + e;
    }
    if (t == 32 || (TH == 32 && t == 31)) {
        int o = 0;
        for (int j = 0; j < L; ++j) {
            s_boff[j] = o;
            o += max(2, 1 << (d.kb[j] + d.nb[j]));  // 16-byte aligned
        }
        s_boff[L] = o;
        s_mx = 0u;
    }
    // this thread's parts
    const int64_t inlo = __ldg(reinterpret_cast<const int64_t *>(d.lo) + t);
    const int64_t outlo = __ldg(reinterpret_cast<const int64_t *>(d.lo) + TH + t);
    const int16_t *rowlo = reinterpret_cast<const int16_t *>(d.lo + 16 * TH) + t;
    __syncthreads();
    float2 *Bs = reinterpret_cast<float2 *>(ch_raw);
    float2 *X0 = Bs + s_boff[L], *X1 = X0 + (int64_t(1) << d.tmax);
    if (t == 0) {
        int ec = 0;
        for (int q = 0; q <= L; ++q) ec += s_E[q];
        s_sc = pow2f(-s_e[0]);
        if (ob == 0) d.EC[inst] = ec;
    }
    for (int j = 0; j < L; ++j) {
        const int kn = 1 << (d.kb[j] + d.nb[j]);
        const float2 *src = d.B[j] + int64_t(s_tab[1 + j]) * kn;
        const float sb = pow2f(-s_e[1 + j]);
        // column n in the kernel's order (its bit b: B's n bit nperm[b])
        for (int e = t; e < kn; e += TH) {
            const int n = e >> d.kb[j];
            int m = 0;
            for (int b = 0; b < d.nb[j]; ++b) m |= ((n >> b) & 1) << d.nperm[j][b];
            const float2 v = __ldg(src + ((m << d.kb[j]) | (e & ((1 << d.kb[j]) - 1))));
            Bs[s_boff[j] + e] = make_float2(v.x * sb, v.y * sb);
        }
    }
    const int64_t n_o = int64_t(1) << d.no;
    const int a = s_tab[0];
    const bool pair_in = d.tin > 0 && d.in_pos[0] == 0, pair_out = tout > 0 && d.out_pos[0] == 0;
    uint32_t lmax = 0u;
    for (int64_t o = ob; o < n_o; o += d.oblocks) {
        // the tile's place in A_1 and C_L: a lane per outside bit
        int64_t abase, cbase;
        {
            uint64_t in = 0, out = 0;
            for (int b = lane; b < d.no; b += 32)
                if ((o >> b) & 1) {
                    in |= uint64_t(1) << d.o_in[b];
                    out |= uint64_t(1) << d.o_out[b];
                }
            const uint32_t il = __reduce_or_sync(0xffffffffu, uint32_t(in)), ih = __reduce_or_sync(0xffffffffu, uint32_t(in >> 32));
            const uint32_t ol = __reduce_or_sync(0xffffffffu, uint32_t(out)), oh = __reduce_or_sync(0xffffffffu, uint32_t(out >> 32));
            abase = int64_t(a) * d.sA + int64_t((uint64_t(ih) << 32) | il);
            cbase = inst * d.sC + int64_t((uint64_t(oh) << 32) | ol);
        }
        // 1. the A_1 tile
        if (pair_in) {
            for (int u = t, i = 0; u < (1 << d.tin) / 2; u += TH, ++i) {
                const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(X0 + swz(2 * u)));
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(d.A + abase + inlo + d.inhi[i])
                             : "memory");
            }
            asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        } else {
            for (int e = t; e < (1 << d.tin); e += TH) {
                int64_t off = 0;
                for (int b = 0; b < d.tin; ++b) off += int64_t((e >> b) & 1) << d.in_pos[b];
                X0[swz(e)] = d.A[abase + off];
            }
        }
        __syncthreads();
        // 2. B_1 .. B_L
        float2 *xi = X0, *xo = X1;
        for (int j = 0; j < L; ++j) {
            StepView v;
            v.B = Bs + s_boff[j];
            v.cpos = d.cpos[j];
            v.col = d.col[j];
            v.pairs = d.nb[j] > 0 && d.cpos[j][0] == 0;
            v.rowhi = d.rowhi[j];
            v.kb = d.kb[j];
            v.nb = d.nb[j];
            v.rbits = d.tb[j] - d.nb[j];
            v.rowlo = __ldg(rowlo + j * TH);
            const bool wide = (1 << v.rbits) >= TH;
            const int kn = wide ? 8 * v.kb + v.nb : -1;
            switch (kn) {
                case 8: step_regs<1, 0>(v, xi, xo, t, TH); break;
                case 9: step_regs<1, 1>(v, xi, xo, t, TH); break;
                case 10: step_regs<1, 2>(v, xi, xo, t, TH); break;
                case 11: step_regs<1, 3>(v, xi, xo, t, TH); break;
                case 16: step_regs<2, 0>(v, xi, xo, t, TH); break;
                case 17: step_regs<2, 1>(v, xi, xo, t, TH); break;
                case 18: step_regs<2, 2>(v, xi, xo, t, TH); break;
                case 24: step_regs<3, 0>(v, xi, xo, t, TH); break;
                case 25: step_regs<3, 1>(v, xi, xo, t, TH); break;
                default:
                    switch (v.kb) {
                        case 0: step_cols<0>(v, xi, xo, t, TH); break;
                        case 1: step_cols<1>(v, xi, xo, t, TH); break;
                        case 2: step_cols<2>(v, xi, xo, t, TH); break;
                        case 3: step_cols<3>(v, xi, xo, t, TH); break;
                        case 4: step_cols<4>(v, xi, xo, t, TH); break;
                        default: step_long(v, xi, xo, t, TH); break;
                    }
            }
            __syncthreads();
            float2 *tmp = xi;
            xi = xo;
            xo = tmp;
        }
        // 3. scale and write the C_L tile
        const float sc = s_sc;
        if (pair_out) {
            for (int u = t, i = 0; u < (1 << tout) / 2; u += TH, ++i) {
                float4 v = *reinterpret_cast<const float4 *>(xi + swz(2 * u));
                v = make_float4(v.x * sc, v.y * sc, v.z * sc, v.w * sc);
                *reinterpret_cast<float4 *>(d.C + cbase + outlo + d.outhi[i]) = v;
                lmax = max(lmax, __float_as_uint(fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)))));
            }
        } else {
            for (int e = t; e < (1 << tout); e += TH) {
                int64_t off = 0;
                for (int b = 0; b < tout; ++b) off += int64_t((e >> b) & 1) << d.out_pos[b];
                const float2 u = xi[swz(e)];
                const float2 v = make_float2(u.x * sc, u.y * sc);
                d.C[cbase + off] = v;
                lmax = max(lmax, __float_as_uint(fmaxf(fabsf(v.x), fabsf(v.y))));
            }
        }
        __syncthreads();  // the buffers are rewritten for the next tile
    }
    if (d.mxC) {
        const uint32_t wmax = __reduce_max_sync(0xffffffffu, lmax);
        if (lane == 0 && wmax) atomicMax(&s_mx, wmax);
        __syncthreads();
        if (t == 0 && s_mx) ch_record_max(d.mxC + inst, s_mx);
    }
}

}  // namespace

size_t chain_smem_bytes(const ChainDesc &d) {
    size_t b = 0;
    for (int j = 0; j < d.L; ++j) {
        const size_t kn = size_t(1) << (d.kb[j] + d.nb[j]);
        b += kn < 2 ? 2 : kn;  // 16-byte aligned
    }
    b += 2 * (size_t(1) << d.tmax);
    return b * sizeof(float2);
}

cudaError_t init_chain_kernel() {
    return cudaFuncSetAttribute(k_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, CH_MAX_SMEM);
}

cudaError_t launch_chain(ChainDesc d, cudaStream_t s) {
    if (d.L < 1 || d.L > CH_MAXL || d.tmax > CH_MAXT || d.no > CH_MAXO) return cudaErrorInvalidValue;
    const size_t smem = chain_smem_bytes(d);
    if (smem > size_t(CH_MAX_SMEM)) return cudaErrorInvalidValue;
    // a tile a block, two where that still leaves several blocks for each of
    // the three that fit an SM
    const int64_t n_o = int64_t(1) << d.no;
    d.oblocks = n_o >= 2 && d.n_inst * n_o >= 4096 ? n_o / 2 : n_o;
    const int64_t blocks = d.n_inst * d.oblocks;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    k_chain<<<dim3((unsigned)blocks), d.threads, smem, s>>>(d);
    return cudaGetLastError();
}

}  // namespace tnk
