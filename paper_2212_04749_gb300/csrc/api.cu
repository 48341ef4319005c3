// C ABI of the contraction library (declared in include/tn.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <tuple>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/tn.h"
#include "kernels.cuh"
#include "plan.hpp"

namespace {

thread_local std::string g_err;

int set_err(int code, const std::string &msg) {
    g_err = msg;
    return code;
}

#define CU(call)                                                                              \
    do {                                                                                      \
        cudaError_t e_ = (call);                                                              \
        if (e_ != cudaSuccess)                                                                \
            return set_err(TN_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));     \
    } while (0)

struct PlanObj {
    tnp::Plan P;
    uint8_t *ws = nullptr;
    size_t ws_bytes = 0;
    std::vector<tnk::StepDesc> desc;  // per step
    struct alignas(64) AMap {
        CUtensorMap map;
        bool ok;
    };
    std::vector<AMap> amap;           // per step: TMA descriptor of A (tensor-core steps)
    std::vector<tnk::ChainDesc> chain_desc;  // per fused chain
    int32_t *err_flag = nullptr;      // device word for bounded waits
    bool tc_fp32 = true;              // FP32 steps take the tensor cores where they may
    bool tc_resident_b = true;        // tensor-core GEMM keeps B in shared memory where it fits
    bool tc_pair = true;              // tensor-core GEMM: column-tile pairs (N = 256 MMAs) where packed B allows
    bool profile = false;
    std::vector<cudaEvent_t> ev;          // pool, two per profiled launch
    std::vector<int> ev_step;             // step of each recorded pair
    size_t ev_used = 0;
    std::vector<int32_t> step_kernel;     // kernel family each step ran last (tn_plan_step_times)
    std::vector<int32_t> step_form;       // TN_FORM_* each step ran last
    std::vector<int32_t> config_override; // per step: -1 plan choice, else a configuration (tn.h)
    // per fused chain: run as one kernel (1), as its steps (0), or not chosen
    // (-1: one kernel, unless all its steps are small: those share the merged
    // launches, which cost less than a kernel of their own)
    std::vector<int8_t> chain_on;
    std::vector<uint8_t> chain_small;     // all steps of the chain are small
    int chain_state(int c) const { return c < (int)chain_on.size() ? chain_on[c] : -1; }
    bool chain_enabled(int c) const { return c >= 0 && chain_state(c) != 0; }
    bool chain_fused(int c) const {
        if (c < 0) return false;
        if (!P.opt.fuse)  // not asked for: not where the caller chose a step's kernel
            for (int s : P.chains[c].steps)
                if (s < (int)pinned.size() && pinned[s]) return false;
        return chain_state(c) > 0 || (chain_state(c) < 0 && !(merge_small && chain_small[c]));
    }
    int reported_chains() const { return P.opt.fuse ? (int)P.chains.size() : 0; }
    struct GraphKey {
        int precision;
        int64_t lo, hi;
        const double *amps;
        bool operator<(const GraphKey &o) const {
            return std::tie(precision, lo, hi, amps) < std::tie(o.precision, o.lo, o.hi, o.amps);
        }
    };
    // Launch order of the steps that a slice batch of one recompute level
    // runs (64: every step).
    struct Sched {
        struct Item {
            int step;   // group < 0: this step's launch (a fused chain's last step: the chain)
            int group;  // else: the small steps of groups[group], one launch
        };
        std::vector<Item> items;
        std::vector<tnk::SmallArgs> groups;
    };
    std::map<int, Sched> scheds;  // by level; dropped with the graphs
    bool merge_small = true;                      // small steps run together (off while the autotuner times them singly)
    std::vector<uint8_t> pinned;                  // per step: the caller chose its kernel (tn_plan_set_config)
    std::vector<uint8_t> apart;                   // per step: the autotuner times it (with a mask), so it merges with none
    std::map<GraphKey, cudaGraphExec_t> graphs;  // captured tn_contract launch sequences
    cudaStream_t cap_stream = nullptr;           // private stream the sequences are captured on
    void drop_graphs() {
        for (auto &kv : graphs) cudaGraphExecDestroy(kv.second);
        graphs.clear();
        scheds.clear();
    }
    int64_t last_batches = 0;
};

template <class T>
T *at(PlanObj *o, int64_t off) {
    return reinterpret_cast<T *>(o->ws + off);
}

// A step's shape as the dispatch sees it: a descriptor without addresses
// (maxima and packed B only present or absent).
tnk::StepDesc shape_desc(const PlanObj *o, const tnp::Step &st) {
    static uint32_t present;
    const tnp::Plan &P = o->P;
    const tnp::Node &nd = P.nodes[st.node], &B = P.nodes[st.b];
    tnk::StepDesc d;
    std::memset(&d, 0, sizeof(d));
    d.mb = st.mb;
    d.kb = st.kb;
    d.nb = st.nb;
    d.nInst = nd.n_inst;
    d.nInstB = d.packBn = B.n_inst;
    d.n_groups = st.n_groups;
    d.max_group = (int32_t)st.max_group;
    d.n_ctab = (int64_t)st.col_tiles.size();
    d.n_ptab = st.n_pair_tiles;
    if (P.opt.rescale) d.mxA = d.mxB = d.mxC = &present;
    if (P.bpack32_bytes > 0) d.bpack = reinterpret_cast<uint8_t *>(&present);
    d.bpack_bytes = P.bpack_bytes;
    d.bpack32_bytes = P.bpack32_bytes;
    d.tc_fp32 = o->tc_fp32 ? 1 : 0;
    d.tc_resident_b = o->tc_resident_b ? 1 : 0;
    d.tc_pair = o->tc_pair ? 1 : 0;
    return d;
}

void build_descs(PlanObj *o) {
    tnp::Plan &P = o->P;
    o->desc.clear();
    for (const tnp::Step &st : P.steps) {
        const tnp::Node &nd = P.nodes[st.node];
        const tnp::Node &A = P.nodes[st.a], &B = P.nodes[st.b];
        tnk::StepDesc d = shape_desc(o, st);
        d.A = at<const float2>(o, A.buf.data);
        d.B = at<const float2>(o, B.buf.data);
        d.C = at<float2>(o, nd.buf.data);
        d.sA = int64_t(1) << A.rank;
        d.sB = int64_t(1) << B.rank;
        d.sC = int64_t(1) << nd.rank;
        const bool a_left = (st.a == nd.left);
        const int32_t *sig = at<const int32_t>(o, nd.buf.sig);
        const int32_t *out = at<const int32_t>(o, nd.buf.out);
        d.sigA = a_left ? sig : sig + nd.n_sig;
        d.sigB = a_left ? sig + nd.n_sig : sig;
        d.outA = a_left ? out : out + nd.n_out;
        d.outB = a_left ? out + nd.n_out : out;
        d.nOutA = A.n_out;
        d.nOutB = B.n_out;
        d.nOut = nd.n_out;
        d.EA = at<const int32_t>(o, A.buf.E);
        d.EB = at<const int32_t>(o, B.buf.E);
        d.EC = at<int32_t>(o, nd.buf.E);
        const bool rs = P.opt.rescale != 0;
        d.mxA = rs ? at<const uint32_t>(o, A.buf.mx) : nullptr;
        d.mxB = rs ? at<const uint32_t>(o, B.buf.mx) : nullptr;
        d.mxC = rs ? at<uint32_t>(o, nd.buf.mx) : nullptr;
        for (int j = 0; j < st.mb; ++j) {
            d.pAm[j] = st.pAm[j];
            d.pCm[j] = st.pCm[j];
        }
        for (int j = 0; j < st.nb; ++j) {
            d.pBn[j] = st.pBn[j];
            d.pCn[j] = st.pCn[j];
        }
        d.gfirst = at<const int64_t>(o, st.off_groups);
        d.ctab = at<const int64_t>(o, st.off_col_tiles);
        d.trec = at<const int4>(o, st.off_tile_rec);
        d.ptab = st.n_pair_tiles > 0 ? at<const int2>(o, st.off_pair_tab) : nullptr;
        d.instab = at<const int2>(o, st.off_inst_ab);
        d.bpack = P.bpack32_bytes > 0 ? at<uint8_t>(o, P.off_bpack) : nullptr;
        o->desc.push_back(d);
    }
    // fused chains
    o->chain_desc.clear();
    for (const tnp::Chain &c : P.chains) {
        tnk::ChainDesc cd;
        std::memset(&cd, 0, sizeof(cd));
        const int L = (int)c.steps.size();
        const tnp::Step &s1 = P.steps[c.steps[0]], &sL = P.steps[c.steps[L - 1]];
        const tnp::Node &A1 = P.nodes[s1.a], &CL = P.nodes[sL.node];
        const bool rs = P.opt.rescale != 0;
        cd.A = at<const float2>(o, A1.buf.data);
        cd.C = at<float2>(o, CL.buf.data);
        cd.sA = int64_t(1) << A1.rank;
        cd.sC = int64_t(1) << CL.rank;
        cd.mxA = rs ? at<const uint32_t>(o, A1.buf.mx) : nullptr;
        cd.mxC = rs ? at<uint32_t>(o, CL.buf.mx) : nullptr;
        cd.EA = at<const int32_t>(o, A1.buf.E);
        cd.EC = at<int32_t>(o, CL.buf.E);
        cd.tab = at<const int32_t>(o, c.off_tab);
        cd.lo = at<const unsigned char>(o, c.off_lo);
        cd.threads = c.threads;
        static_assert(tnk::CH_ROUNDS == tnp::CHAIN_ROUNDS && tnk::CH_MAXT == tnp::CHAIN_MAX_TILE_BITS &&
                          tnk::CH_MAXL == tnp::CHAIN_MAX_STEPS, "the planner's chain is the kernel's");
        for (int i = 0; i < tnk::CH_ROUNDS; ++i) {
            for (size_t b = 0; b + 1 < c.in_pos.size(); ++b)
                if (((int64_t(i) * c.threads) >> b) & 1) cd.inhi[i] += int64_t(1) << c.in_pos[b + 1];
            for (size_t b = 0; b + 1 < c.out_pos.size(); ++b)
                if (((int64_t(i) * c.threads) >> b) & 1) cd.outhi[i] += int64_t(1) << c.out_pos[b + 1];
        }
        cd.n_inst = CL.n_inst;
        cd.L = L;
        cd.tin = c.tin;
        cd.no = c.no;
        cd.tmax = c.tin;
        for (int j = 0; j < L; ++j) {
            const tnp::Step &st = P.steps[c.steps[j]];
            const tnp::Node &B = P.nodes[st.b];
            cd.B[j] = at<const float2>(o, B.buf.data);
            cd.mxB[j] = rs ? at<const uint32_t>(o, B.buf.mx) : nullptr;
            cd.EB[j] = at<const int32_t>(o, B.buf.E);
            cd.kb[j] = st.kb;
            cd.nb[j] = st.nb;
            cd.tb[j] = c.tbits[j];
            cd.tmax = std::max(cd.tmax, c.tbits[j]);
            // columns in the kernel's order: the n bit at the output's lowest
            // address bit first, if there is one
            const size_t nb = c.cpos[j].size();
            for (size_t b = 0; b < nb; ++b) cd.nperm[j][b] = (int8_t)b;
            for (size_t b = 1; b < nb; ++b)
                if (c.cpos[j][b] == 0) std::swap(cd.nperm[j][0], cd.nperm[j][b]);
            for (size_t b = 0; b < nb; ++b) cd.cpos[j][b] = c.cpos[j][cd.nperm[j][b]];
            for (int i = 0; i < tnk::CH_ROUNDS; ++i) {
                int r = 0, n = 0;
                for (size_t b = 0; b < c.rpos[j].size(); ++b)
                    if (((int64_t(i) * c.threads) >> b) & 1) r |= 1 << c.rpos[j][b];
                for (size_t b = 0; b < nb && b < 4; ++b) n |= ((i >> b) & 1) << cd.cpos[j][b];
                cd.rowhi[j][i] = (int16_t)tnp::chain_swz(r);
                cd.col[j][i] = (int16_t)tnp::chain_swz(n);
            }
        }
        for (int b = 0; b < c.tin; ++b) cd.in_pos[b] = c.in_pos[b];
        for (size_t b = 0; b < c.out_pos.size(); ++b) cd.out_pos[b] = c.out_pos[b];
        for (int b = 0; b < c.no; ++b) {
            cd.o_in[b] = c.o_in_pos[b];
            cd.o_out[b] = c.o_out_pos[b];
        }
        o->chain_desc.push_back(cd);
    }
    // TMA descriptors of the A operands, for every step the tensor-core
    // kernel can take (it may be chosen at run time)
    o->amap.assign(P.steps.size(), PlanObj::AMap{});
    for (size_t s = 0; s < P.steps.size(); ++s) {
        const tnk::StepDesc &d = o->desc[s];
        o->amap[s].ok = tnk::gemm_tc_supports(d) &&
                        tnk::make_a_map(d, P.nodes[P.steps[s].a].n_inst, &o->amap[s].map) == cudaSuccess;
    }
}

// The steps as small.cu sees them (those that are not small stay empty).
std::vector<tnk::SmallDesc> small_descs(const PlanObj *o) {
    static_assert(sizeof(tnk::SmallDesc) == tnp::SMALL_DESC_BYTES, "room in the workspace");
    std::vector<tnk::SmallDesc> v(o->P.steps.size());
    for (size_t s = 0; s < v.size(); ++s) {
        const tnk::StepDesc &d = o->desc[s];
        tnk::SmallDesc &r = v[s];
        std::memset(&r, 0, sizeof(r));
        if (!o->P.steps[s].small) continue;
        r.A = d.A;
        r.B = d.B;
        r.C = d.C;
        r.instab = d.instab;
        r.EA = d.EA;
        r.EB = d.EB;
        r.EC = d.EC;
        r.mxA = d.mxA;
        r.mxB = d.mxB;
        r.mxC = d.mxC;
        r.sA = d.sA;
        r.sB = d.sB;
        r.sC = d.sC;
        r.kb = (int8_t)d.kb;
        r.nb = (int8_t)d.nb;
        r.mnb = (int8_t)(d.mb + d.nb);
        r.outputs = (int32_t)(d.nInst << (d.mb + d.nb));
        for (int j = 0; j < d.nb; ++j) r.pC[j] = d.pCn[j];
        for (int j = 0; j < d.mb; ++j) r.pC[d.nb + j] = d.pCm[j];
    }
    return v;
}

// Configurations (tn.h): 0, 1 per-row kernel (schedule 0, 1); 2, 3 grouped
// GEMM (schedule 0, 1).
bool config_allowed(const tnp::Step &S, int c) {
    if (c < 0 || c >= TN_NCONFIG) return false;
    return c >= 2 || (S.nb <= 4 && S.kb + S.nb <= 8);
}

// The configuration that the plan takes by itself.
int own_config(const tnp::Step &S) { return S.kernel == 0 ? 0 : 2; }

int effective_config(const PlanObj *o, int s) {
    if (s < (int)o->config_override.size() && o->config_override[s] >= 0) return o->config_override[s];
    return own_config(o->P.steps[s]);
}

// The slice instance of node nd that low slice bits sigma select: the bits
// of its own batched edges, compressed.
int64_t slice_instance(const tnp::Node &nd, int64_t sigma) {
    int64_t r = 0;
    for (size_t j = 0; j < nd.slices_low.size(); ++j) r |= ((sigma >> nd.slices_low[j]) & 1) << j;
    return r;
}

// Narrow a step to the output instances of one slice: the groups that hold
// them (a group that reaches beyond them is computed whole; its other
// instances are then never read).
void apply_window(const PlanObj *o, const tnp::Step &S, int64_t sigma, tnk::StepDesc &d) {
    const tnp::Node &nd = o->P.nodes[S.node], &B = o->P.nodes[S.b];
    const int64_t i0 = slice_instance(nd, sigma) * nd.n_out, i1 = i0 + nd.n_out;
    const auto &gf = S.group_first;
    const int64_t g0 = std::upper_bound(gf.begin(), gf.end(), i0) - gf.begin() - 1;
    const int64_t g1 = std::lower_bound(gf.begin(), gf.end(), i1) - gf.begin();
    const auto &ct = S.col_tiles;
    const int64_t t0 = std::lower_bound(ct.begin(), ct.end(), g0 << 20) - ct.begin();
    const int64_t t1 = std::lower_bound(ct.begin(), ct.end(), g1 << 20) - ct.begin();
    d.inst0 = i0;
    d.nInst = nd.n_out;
    d.gfirst += g0;
    d.n_groups = g1 - g0;
    d.trec += t0;
    d.ctab += t0;
    d.n_ctab = t1 - t0;
    d.tile0 = t0;
    if (d.ptab) {
        int64_t p0 = 0, p1 = 0;
        for (int64_t g = 0; g < g1; ++g) {
            const int64_t n = gf[g + 1] - gf[g];
            (g < g0 ? p0 : p1) += n + (n & 1);
        }
        d.ptab += p0;
        d.ptile0 = p0;
        d.n_ptab = p1;
    }
    d.packB0 = slice_instance(B, sigma) * B.n_out;
    d.packBn = B.n_out;
}

// The kernel (TN_FORM_*) of a step under configuration cfg, and its schedule
// (d.sched).  ruled: nobody chose the configuration; few: an output per
// thread is not allowed (0), where it is the faster under every configuration
// (1), also where only the plan's own, cfg, is slower (2); map_ok: A has a TMA descriptor (FP32; the other
// precisions fail without one).
int step_form(tnk::StepDesc &d, int cfg, bool ruled, int precision, int few, bool map_ok) {
    d.sched = cfg & 1;
    const bool skinny = tnk::step_skinny_takes(d);
    const bool on_tc = cfg >= 2 && precision != TN_FP32 && tnk::gemm_tc_supports(d) && !skinny;
    if (few && tnk::step_few_takes(d, on_tc, few == 2)) return TN_FORM_FEW;
    if (cfg < 2) return tnk::step_row_narrow(d) ? TN_FORM_NARROW : TN_FORM_ROW;
    if (skinny) return TN_FORM_SKINNY;  // few outputs per instance and a long K (e.g. the root)
    if (on_tc) {
        if (ruled) d.sched = tnk::tc_rule_schedule(d);
        return d.tc_resident_b && tnk::tc_dictionary_chunks(d) == 0 && tnk::tc_resident_b_chunks(d) == 0 &&
                       tnk::step_narrow_takes(d, false)
                   ? TN_FORM_NARROW
                   : TN_FORM_TC;
    }
    if (precision == TN_FP32 && map_ok && tnk::tc_fp32_takes(d)) return TN_FORM_TC_FP32;
    if (tnk::step_outer_takes(d)) return TN_FORM_OUTER;
    return tnk::step_narrow_takes(d, true) ? TN_FORM_NARROW : TN_FORM_SIMT;
}

// The family (tn_plan_step_times) of a TN_FORM_* under a configuration.
int family_of(int form, int cfg) {
    switch (form) {
        case TN_FORM_ROW: return 0;
        case TN_FORM_NARROW: return cfg < 2 ? 0 : 1;
        case TN_FORM_TC:
        case TN_FORM_TC_FP32: return 2;
        case TN_FORM_CHAIN: return 3;
        case TN_FORM_SMALL: return 4;
        default: return 1;
    }
}

// sigma >= 0: only the output instances of that slice of the pass
int run_step(PlanObj *o, int s, int precision, int64_t sigma, cudaStream_t st) {
    const tnp::Step &S = o->P.steps[s];
    if (o->chain_fused(S.chain)) {  // fused chain: runs whole at its last step
        tnk::ChainDesc c = o->chain_desc[S.chain];
        if (sigma >= 0) {
            const tnp::Node &nd = o->P.nodes[S.node];
            c.inst0 = slice_instance(nd, sigma) * nd.n_out;
            c.n_inst = nd.n_out;
        }
        const cudaError_t e = tnk::launch_chain(c, st);
        if (e != cudaSuccess)
            return set_err(TN_ECUDA, "fused chain at step " + std::to_string(s) + ": " + cudaGetErrorString(e));
        return TN_OK;
    }
    const int cfg = effective_config(o, s);
    tnk::StepDesc d = o->desc[s];
    if (sigma >= 0) apply_window(o, S, sigma, d);
    d.tc_fp32 = o->tc_fp32 ? 1 : 0;
    d.tc_resident_b = o->tc_resident_b ? 1 : 0;
    d.tc_pair = o->tc_pair ? 1 : 0;
    const bool chosen = s < (int)o->pinned.size() && o->pinned[s];  // by the caller: runs as it is
    const bool ruled = !(s < (int)o->config_override.size() && o->config_override[s] >= 0);
    const int form = step_form(d, cfg, ruled, precision, chosen ? 0 : (cfg == own_config(S) ? 2 : 1), o->amap[s].ok);
    cudaError_t e;
    switch (form) {
        case TN_FORM_FEW: e = tnk::launch_step_few(d, st); break;
        case TN_FORM_ROW: e = tnk::launch_step_row(d, st); break;
        case TN_FORM_NARROW: e = cfg < 2 ? tnk::launch_step_row(d, st) : tnk::launch_step_narrow(d, st); break;
        case TN_FORM_SKINNY: e = tnk::launch_step_skinny(d, st); break;
        case TN_FORM_OUTER: e = tnk::launch_step_outer(d, st); break;
        case TN_FORM_SIMT: e = tnk::launch_step_gemm_simt(d, st); break;
        default:
            e = o->amap[s].ok ? tnk::launch_step_gemm_tc(d, &o->amap[s].map, precision, o->err_flag, st)
                              : cudaErrorInvalidValue;  // its TMA descriptor could not be encoded
    }
    o->step_form[s] = form;
    o->step_kernel[s] = family_of(form, cfg);
    if (e != cudaSuccess)
        return set_err(TN_ECUDA, "step " + std::to_string(s) + ": " + cudaGetErrorString(e));
    return TN_OK;
}

int run_group(PlanObj *o, tnk::SmallArgs g, cudaStream_t st) {
    g.descs = at<const tnk::SmallDesc>(o, o->P.off_small);
    for (int j = 0; j < g.n_steps; ++j) {
        o->step_form[g.step[j]] = TN_FORM_SMALL;
        o->step_kernel[g.step[j]] = 4;
    }
    const cudaError_t e = tnk::launch_small(g, st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("small steps: ") + cudaGetErrorString(e));
    return TN_OK;
}

// Whether step s may share a launch with other small steps.
bool merges(const PlanObj *o, int s) {
    return o->merge_small && o->P.steps[s].small && !(s < (int)o->pinned.size() && o->pinned[s]) &&
           !(s < (int)o->apart.size() && o->apart[s]);
}

// Launch order for a slice batch of recompute level lv (64: every step).
// The steps keep the plan's order except that small ones move: they wait
// until a step that does not merge needs one of them, and then every small
// step whose operands exist runs in the same launch, in phases.  Two steps
// keep their order where the later reads what the earlier writes, or writes
// memory that the earlier reads or writes (the workspace gives a slot to
// another node after its last reader in the plan's order).
PlanObj::Sched make_schedule(const PlanObj *o, int lv) {
    PlanObj::Sched R;
    const tnp::Plan &P = o->P;
    struct Node {
        int step, write;
        std::vector<int> reads;
        bool small;
    };
    std::vector<Node> L;
    for (int s = 0; s < (int)P.steps.size(); ++s) {
        const tnp::Step &S = P.steps[s];
        if (S.level > lv) continue;
        Node n{s, S.node, {}, false};
        if (o->chain_fused(S.chain)) {
            if (!S.chain_last) continue;
            const tnp::Chain &c = P.chains[S.chain];
            n.reads.push_back(P.steps[c.steps[0]].a);
            for (int q : c.steps) n.reads.push_back(P.steps[q].b);
        } else {
            n.reads = {S.a, S.b};
            n.small = merges(o, s);
        }
        L.push_back(n);
    }
    const int nl = (int)L.size();
    auto overlap = [&](int u, int v) {
        const tnp::Node &x = P.nodes[u], &y = P.nodes[v];
        return x.buf.data < y.buf.data + y.n_inst * (int64_t(8) << y.rank) &&
               y.buf.data < x.buf.data + x.n_inst * (int64_t(8) << x.rank);
    };
    std::vector<std::vector<int>> after(nl);  // edges to later items
    std::vector<int> open(nl, 0);             // unfinished items before
    for (int q = 0; q < nl; ++q)
        for (int p = 0; p < q; ++p) {
            bool dep = overlap(L[q].write, L[p].write);
            for (int r : L[q].reads) dep = dep || r == L[p].write;
            for (int r : L[p].reads) dep = dep || overlap(L[q].write, r);
            if (dep) {
                after[p].push_back(q);
                ++open[q];
            }
        }
    std::vector<char> done(nl, 0);
    auto finish = [&](int q) {
        done[q] = 1;
        for (int t : after[q]) --open[t];
    };
    int left = nl, next_big = 0;
    while (left > 0) {
        while (next_big < nl && (done[next_big] || L[next_big].small)) ++next_big;
        if (next_big < nl && open[next_big] == 0) {
            R.items.push_back({L[next_big].step, -1});
            finish(next_big);
            --left;
            continue;
        }
        tnk::SmallArgs g;
        std::memset(&g, 0, sizeof(g));
        int last = -1;
        while (g.n_phases < tnk::SMALL_MAX_PHASES && g.n_steps < tnk::SMALL_MAX_STEPS) {
            std::vector<int> ready;
            int64_t outputs = 0;
            for (int q = 0; q < nl && g.n_steps + (int)ready.size() < tnk::SMALL_MAX_STEPS; ++q)
                if (!done[q] && L[q].small && open[q] == 0) {
                    ready.push_back(q);
                    const tnp::Step &S = P.steps[L[q].step];
                    outputs += P.nodes[S.node].n_inst << (S.mb + S.nb);
                }
            if (ready.empty()) break;
            // lanes per output: as many as leave the phase within 8192 threads
            int lanes = 0;
            while (lanes < 5 && (outputs << (lanes + 1)) <= 8192) ++lanes;
            int64_t warps = 0;
            for (int q : ready) {
                const tnp::Step &S = P.steps[L[q].step];
                const int lg = std::min(lanes, std::max(S.kb - 1, 0));
                // a warp takes 32 lanes of outputs, four times as many where
                // the step fills the cluster's 256 warps four times over
                const int64_t w = (((P.nodes[S.node].n_inst << (S.mb + S.nb)) << lg) + 31) / 32;
                const bool four = w >= 1024;
                g.four[g.n_steps] = four;
                warps += four ? (w + 3) / 4 : w;
                g.step[g.n_steps] = (uint16_t)L[q].step;
                g.lanes_log2[g.n_steps] = (uint8_t)lg;
                g.wend[g.n_steps] = (int32_t)warps;
                last = std::max(last, L[q].step);
                ++g.n_steps;
            }
            for (int q : ready) finish(q);
            left -= (int)ready.size();
            g.max_warps = std::max<int32_t>(g.max_warps, (int32_t)std::min<int64_t>(warps, 1 << 20));
            g.phase_end[g.n_phases++] = (uint16_t)g.n_steps;
        }
        if (g.n_steps == 1) {
            R.items.push_back({last, -1});
        } else {
            R.items.push_back({last, (int)R.groups.size()});
            R.groups.push_back(g);
        }
    }
    return R;
}

const PlanObj::Sched &schedule(PlanObj *o, int lv) {
    auto it = o->scheds.find(lv);
    if (it == o->scheds.end()) it = o->scheds.emplace(lv, make_schedule(o, lv)).first;
    return it->second;
}

// Cost-model features of step s under configuration c (tn.h, TN_NFEAT).
void step_features(const PlanObj *o, int s, int precision, int c, float *f) {
    const tnp::Plan &P = o->P;
    const tnp::Step &S = P.steps[s];
    const tnp::Node &nd = P.nodes[S.node], &A = P.nodes[S.a], &B = P.nodes[S.b];
    auto lg = [](double x) { return float(std::log2(x > 1.0 ? x : 1.0)); };
    auto run = [](const std::vector<int8_t> &pos) {
        int j = 0;
        while (j < (int)pos.size() && pos[j] == j) ++j;
        return j;
    };
    int crun = 0;  // lowest C address bits held by consecutive m bits
    while (crun < S.mb && S.pCm[crun] == crun) ++crun;
    tnk::StepDesc t = shape_desc(o, S);
    const int form = step_form(t, c, false, precision, c == own_config(S) ? 2 : 1, true);
    const bool gemm = c >= 2, tc = form == TN_FORM_TC || form == TN_FORM_TC_FP32;
    const double ng = double(S.n_groups > 0 ? S.n_groups : 1);
    int i = 0;
    f[i++] = S.mb / 32.f;
    f[i++] = S.kb / 32.f;
    f[i++] = S.nb / 32.f;
    f[i++] = A.rank / 32.f;
    f[i++] = B.rank / 32.f;
    f[i++] = lg(double(nd.n_inst)) / 32.f;
    f[i++] = lg(double(A.n_inst)) / 32.f;
    f[i++] = lg(double(B.n_inst)) / 32.f;
    f[i++] = lg(ng) / 32.f;
    f[i++] = lg(double(nd.n_inst) / ng * std::ldexp(1.0, S.nb)) / 32.f;
    f[i++] = run(S.pAm) / 32.f;
    f[i++] = run(S.pAk) / 32.f;
    f[i++] = run(S.pBk) / 32.f;
    f[i++] = run(S.pBn) / 32.f;
    f[i++] = crun / 32.f;
    f[i++] = lg(S.flops) / 64.f;
    f[i++] = lg(S.bytes) / 64.f;
    f[i++] = precision == TN_TF32 ? 1.f : 0.f;
    f[i++] = precision == TN_BF16X3 ? 1.f : 0.f;
    f[i++] = gemm ? 0.f : 1.f;
    f[i++] = tc ? 1.f : 0.f;
    f[i++] = gemm && !tc ? 1.f : 0.f;
    f[i++] = float(c & 1);
    f[i++] = lg(double(nd.n_inst) * std::ldexp(1.0, S.mb)) / 64.f;
}

void start_launches(PlanObj *o) {
    const tnp::Plan &P = o->P;
    o->step_kernel.resize(P.steps.size(), -1);
    o->step_form.resize(P.steps.size(), -1);
    for (size_t s = 0; s < P.steps.size(); ++s)
        if (o->chain_fused(P.steps[s].chain)) {
            o->step_form[s] = TN_FORM_CHAIN;
            o->step_kernel[s] = 3;
        }
    o->ev_used = 0;
    o->ev_step.clear();
}

// Estimated time (us) of a pass over the steps of level <= lv (-1: none),
// of whole steps or of those that hold one slice's instances: a launch costs
// about 5 us whatever it computes, a merged one 5 and 2 a phase, and the
// other steps their bytes or flops at about the rates that they reach.
double pass_us(PlanObj *o, int precision, int lv, bool narrow) {
    if (lv < 0) return 0.0;
    const tnp::Plan &P = o->P;
    const PlanObj::Sched &order = schedule(o, lv);
    double t = 10.0;  // maxima cleared, leaves filled
    for (const PlanObj::Sched::Item &it : order.items) {
        if (it.group >= 0) {
            t += 5.0 + 2.0 * order.groups[it.group].n_phases;
            continue;
        }
        const tnp::Step &S = P.steps[it.step];
        const tnp::Node &nd = P.nodes[S.node];
        double bytes = S.bytes, flops = S.flops, rate = 60e6;  // flops a us
        if (o->chain_fused(S.chain)) {
            const tnp::Chain &c = P.chains[S.chain];
            const tnp::Node &A = P.nodes[P.steps[c.steps[0]].a];
            bytes = 8.0 * (std::ldexp(double(A.n_inst), A.rank) + std::ldexp(double(nd.n_inst), nd.rank));
            flops = 0.0;
            for (int q : c.steps) flops += P.steps[q].flops;
        } else if (effective_config(o, it.step) >= 2 && !tnk::step_skinny_takes(o->desc[it.step])) {
            if (precision != TN_FP32 && tnk::gemm_tc_supports(o->desc[it.step])) rate = precision == TN_TF32 ? 500e6 : 320e6;
        }
        const double part = narrow ? std::ldexp(1.0, -(int)nd.slices_low.size()) : 1.0;
        t += std::max(5.0, part * std::max(bytes / 6e6, flops / rate));
    }
    return t;
}

// One pass over slice batch b: the steps of level <= lv (64: all), the
// others keep what an earlier pass left.  sigma >= 0: one slice of the batch.
int run_pass(PlanObj *o, int precision, int64_t b, int lv, int64_t sigma, cudaStream_t st) {
    tnp::Plan &P = o->P;
    const auto *jobs = at<const tnk::FillJobD>(o, P.off_fill_jobs);
    const auto *highs = at<const tnk::LeafHighD>(o, P.off_leaf_high);
    const int64_t clear = lv >= 64 ? P.emax_bytes : P.emax_prefix[lv];
    if (clear) CU(cudaMemsetAsync(o->ws + P.off_emax, 0, clear, st));
    cudaError_t e = tnk::launch_fill(jobs, P.n_fill_jobs, highs, b, at<float2>(o, 0), st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("leaf fill: ") + cudaGetErrorString(e));
    const PlanObj::Sched &order = schedule(o, lv);
    for (const PlanObj::Sched::Item &it : order.items) {
        const int s = it.step;
        if (o->profile) {
            while (o->ev.size() < 2 * (o->ev_used + 1)) {
                cudaEvent_t ev;
                CU(cudaEventCreate(&ev));
                o->ev.push_back(ev);
            }
            CU(cudaEventRecord(o->ev[2 * o->ev_used], st));
        }
        // merged small steps compute every slice of the pass
        if (it.group >= 0) {
            if (int rc = run_group(o, order.groups[it.group], st)) return rc;
        } else if (int rc = run_step(o, s, precision, sigma, st)) {
            return rc;
        }
        if (o->profile) {
            CU(cudaEventRecord(o->ev[2 * o->ev_used + 1], st));
            o->ev_step.push_back(s);
            o->ev_used++;
        }
    }
    return TN_OK;
}

// Batches [b_lo, b_hi) in order.  The first batch of the call runs every
// step; batch b > b_lo re-runs only the steps whose sliced edges changed
// from batch b-1 (level <= ctz(b)).  `per_batch(b)` runs after each batch.
template <class F>
int run_batches(PlanObj *o, int precision, int64_t b_lo, int64_t b_hi, cudaStream_t st, F per_batch) {
    start_launches(o);
    for (int64_t b = b_lo; b < b_hi; ++b) {
        const int lv = (b == b_lo) ? 64 : __builtin_ctzll((unsigned long long)b);
        if (int rc = run_pass(o, precision, b, lv, -1, st)) return rc;
        if (int rc = per_batch(b)) return rc;
    }
    o->last_batches = b_hi - b_lo;
    return TN_OK;
}

// Fixed device scratch for tn_contract_static.  In host code this name is a
// host-side stand-in, not a device address: the address comes from
// cudaGetSymbolAddress, looked up once per device.
__device__ __align__(256) unsigned char g_static_scratch[TN_STATIC_SCRATCH_BYTES];

std::mutex g_static_mu;
std::vector<void *> g_static_addr;  // per device ordinal; null until looked up

int static_scratch_address(void **out) {
    int dev = 0;
    CU(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_static_mu);
    if ((int)g_static_addr.size() <= dev) g_static_addr.resize(dev + 1, nullptr);
    if (!g_static_addr[dev]) {
        void *p = nullptr;
        CU(cudaGetSymbolAddress(&p, g_static_scratch));
        g_static_addr[dev] = p;
    }
    *out = g_static_addr[dev];
    return TN_OK;
}

}  // namespace

extern "C" {

const char *tn_last_error(void) { return g_err.c_str(); }

int tn_network(const tn_circuit *circ, int32_t *n_tensors, int32_t *n_edges, int32_t *edge_ends,
               int32_t *out_tensor) {
    tnp::Network net;
    std::string err;
    if (!tnp::build_network(circ, net, err)) return set_err(TN_EINVAL, err);
    if (n_tensors) *n_tensors = net.n_tensors;
    if (n_edges) *n_edges = net.n_edges;
    if (edge_ends)
        for (int e = 0; e < net.n_edges; ++e) {
            edge_ends[2 * e] = net.edge_ends[e][0];
            edge_ends[2 * e + 1] = net.edge_ends[e][1];
        }
    if (out_tensor)
        for (int q = 0; q < net.n_qubits; ++q) out_tensor[q] = net.out_tensor[q];
    g_err.clear();
    return TN_OK;
}

int tn_plan(const tn_circuit *circ, const uint8_t *bits, int64_t k, const int32_t *tree_ssa,
            const int32_t *sliced_edges, int32_t n_sliced, const tn_options *opt, tn_plan_t *out) {
    if (!out) return set_err(TN_EINVAL, "tn_plan: null output handle");
    *out = nullptr;
    std::unique_ptr<PlanObj> o(new PlanObj());
    std::string err;
    int code = TN_OK;
    try {
        if (!tnp::make_plan(circ, bits, k, tree_ssa, sliced_edges, n_sliced, opt, o->P, err, code))
            return set_err(code, err);
    } catch (const std::bad_alloc &) {
        return set_err(TN_ENOMEM, "tn_plan: host allocation failed");
    }
    for (const tnp::Chain &c : o->P.chains) {
        bool all = true;
        for (int q : c.steps) all = all && o->P.steps[q].small;
        o->chain_small.push_back(all ? 1 : 0);
    }
    *out = reinterpret_cast<tn_plan_t>(o.release());
    g_err.clear();
    return TN_OK;
}

int tn_plan_query(tn_plan_t plan, tn_plan_info *info) {
    if (!plan || !info) return set_err(TN_EINVAL, "tn_plan_query: null argument");
    const tnp::Plan &P = reinterpret_cast<PlanObj *>(plan)->P;
    std::memset(info, 0, sizeof(*info));
    info->n_tensors = P.net.n_tensors;
    info->n_edges = P.net.n_edges;
    info->n_nodes = (int32_t)P.nodes.size();
    info->n_steps = (int32_t)P.steps.size();
    info->n_unique = (int32_t)P.k_unique;
    info->n_sliced = (int32_t)P.sliced.size();
    info->slice_batch_log2 = P.m_low;
    info->n_batches = (int32_t)P.n_batches;
    info->max_rank = P.max_rank;
    info->n_static_steps = P.n_static_steps;
    info->flops_ma = P.flops_ma;
    info->flops_sa = P.flops_sa;
    info->flops_exec = P.flops_exec;
    info->bytes_min = P.bytes_min;
    info->workspace_bytes = P.ws_bytes;
    info->peak_tensor_bytes = P.peak_tensor_bytes;
    int64_t up = 0;
    for (const auto &u : P.uploads) up += (int64_t)u.second.size();
    info->upload_bytes = up;
    const PlanObj *po = reinterpret_cast<const PlanObj *>(plan);
    double steps_run = 0;
    for (const tnp::Step &st : P.steps)
        steps_run += (!P.opt.fuse || !po->chain_enabled(st.chain) || st.chain_last) ? st.runs : 0.0;
    info->launches_per_call = (int64_t)steps_run + 2 * P.n_batches;  // + leaf fill and accumulate per batch
    info->n_open = (int32_t)P.open_qubits.size();
    info->n_chains = po->reported_chains();
    info->amps_per_row = int64_t(1) << P.open_qubits.size();
    return TN_OK;
}

int tn_plan_launches(tn_plan_t plan, int64_t *launches) {
    if (!plan || !launches) return set_err(TN_EINVAL, "tn_plan_launches: null argument");
    const PlanObj *o = reinterpret_cast<const PlanObj *>(plan);
    // the first batch runs every step, n_batches >> (l + 1) later ones those of level l and below
    const int64_t nb = o->P.n_batches;
    int64_t n = 2 * nb + (int64_t)make_schedule(o, 64).items.size();
    for (int l = 0; (nb >> (l + 1)) > 0; ++l) n += (nb >> (l + 1)) * (int64_t)make_schedule(o, l).items.size();
    *launches = n;
    g_err.clear();
    return TN_OK;
}

int tn_plan_widths(tn_plan_t plan, int64_t *width_out, int32_t *rank, int32_t *n_slice_vars) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_widths: null plan");
    const tnp::Plan &P = reinterpret_cast<PlanObj *>(plan)->P;
    for (size_t v = 0; v < P.nodes.size(); ++v) {
        if (width_out) width_out[v] = P.nodes[v].n_out;
        if (rank) rank[v] = P.nodes[v].rank;
        if (n_slice_vars) n_slice_vars[v] = (int32_t)P.nodes[v].slices.size();
    }
    return TN_OK;
}

int tn_plan_steps(tn_plan_t plan, tn_step_info *out, int32_t n) {
    if (!plan || (n > 0 && !out)) return set_err(TN_EINVAL, "tn_plan_steps: null argument");
    const tnp::Plan &P = reinterpret_cast<PlanObj *>(plan)->P;
    for (int32_t s = 0; s < n && s < (int32_t)P.steps.size(); ++s) {
        const tnp::Step &st = P.steps[s];
        tn_step_info &r = out[s];
        r.node = st.node;
        r.a = st.a;
        r.b = st.b;
        r.mb = st.mb;
        r.kb = st.kb;
        r.nb = st.nb;
        r.rank_a = P.nodes[st.a].rank;
        r.rank_b = P.nodes[st.b].rank;
        r.level = st.level;
        r.kernel = st.kernel;
        r.n_inst = P.nodes[st.node].n_inst;
        r.n_inst_a = P.nodes[st.a].n_inst;
        r.n_inst_b = P.nodes[st.b].n_inst;
        r.flops = st.flops;
        r.bytes = st.bytes;
        r.runs = st.runs;
        auto run = [](const std::vector<int8_t> &pos) {
            int j = 0;
            while (j < (int)pos.size() && pos[j] == j) ++j;
            return j;
        };
        r.a_run_m = run(st.pAm);
        r.a_run_k = run(st.pAk);
        r.b_run_k = run(st.pBk);
        r.b_run_n = run(st.pBn);
        r.n_groups = st.n_groups;
        r.chain = P.opt.fuse ? st.chain : -1;
        r.chain_last = P.opt.fuse && st.chain_last ? 1 : 0;
        for (int j = 0; j < 40; ++j) r.c_pos_m[j] = j < st.mb ? st.pCm[j] : -1;
        for (int j = 0; j < 24; ++j) r.c_pos_n[j] = j < st.nb ? st.pCn[j] : -1;
        r.max_group = st.max_group;
        r.n_pair_tiles = st.n_pair_tiles;
    }
    return TN_OK;
}

int tn_plan_batch_slices(tn_plan_t plan, int64_t batch, int64_t *slice_ids, int64_t n) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_batch_slices: null plan");
    const tnp::Plan &P = reinterpret_cast<PlanObj *>(plan)->P;
    const int64_t per = int64_t(1) << P.m_low;
    if (batch < 0 || batch >= P.n_batches) return set_err(TN_EINVAL, "tn_plan_batch_slices: batch outside [0, n_batches)");
    if (n < per || !slice_ids)
        return set_err(TN_EINVAL, "tn_plan_batch_slices: need room for " + std::to_string(per) + " slice ids");
    for (int64_t sigma = 0; sigma < per; ++sigma) {
        const int64_t v = batch * per + sigma;  // internal slice index
        int64_t ext = 0;
        for (size_t t = 0; t < P.perm.size(); ++t) ext |= ((v >> t) & 1) << P.perm[t];
        slice_ids[sigma] = ext;
    }
    return TN_OK;
}

int tn_plan_bind(tn_plan_t plan, void *workspace, size_t bytes, void *stream) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_bind: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255))
        return set_err(TN_EINVAL, "tn_plan_bind: workspace must be a 256-byte aligned device pointer");
    if ((int64_t)bytes < o->P.ws_bytes)
        return set_err(TN_ENOMEM, "tn_plan_bind: workspace has " + std::to_string(bytes) + " bytes, plan needs " +
                                      std::to_string(o->P.ws_bytes));
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    CU(tnk::init_kernels());
    CU(tnk::init_chain_kernel());
    CU(tnk::init_simt_kernels());
    CU(tnk::init_small_kernel());
    o->drop_graphs();
    o->ws = static_cast<uint8_t *>(workspace);
    o->ws_bytes = bytes;
    for (auto &u : o->P.uploads) {
        if (u.second.empty()) continue;
        CU(cudaMemcpyAsync(o->ws + u.first, u.second.data(), u.second.size(), cudaMemcpyHostToDevice, st));
    }
    o->err_flag = at<int32_t>(o, o->P.off_scratch);
    CU(cudaMemsetAsync(o->err_flag, 0, 4, st));
    build_descs(o);
    const std::vector<tnk::SmallDesc> small = small_descs(o);
    CU(cudaMemcpyAsync(o->ws + o->P.off_small, small.data(), small.size() * sizeof(tnk::SmallDesc),
                       cudaMemcpyHostToDevice, st));
    CU(cudaStreamSynchronize(st));
    g_err.clear();
    return TN_OK;
}

int tn_contract(tn_plan_t plan, int precision, int64_t batch_lo, int64_t batch_hi, double *amps, void *stream) {
    if (!plan) return set_err(TN_EINVAL, "tn_contract: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (!o->ws) return set_err(TN_ESTATE, "tn_contract: no workspace bound (call tn_plan_bind)");
    if (precision < TN_FP32 || precision > TN_BF16X3) return set_err(TN_EINVAL, "tn_contract: bad precision");
    tnp::Plan &P = o->P;
    if (batch_lo < 0 || batch_hi > P.n_batches || batch_lo > batch_hi)
        return set_err(TN_EINVAL, "tn_contract: batch range outside [0, n_batches)");
    if (P.k == 0 || batch_lo == batch_hi) return TN_OK;
    if (!amps) return set_err(TN_EINVAL, "tn_contract: null amplitude buffer");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const tnp::Node &R = P.nodes[P.root];
    const float2 *root = at<const float2>(o, R.buf.data);
    const int32_t *E = at<const int32_t>(o, R.buf.E);
    const int32_t *uniq = at<const int32_t>(o, P.off_uniq);
    auto enqueue = [&]() {
        return run_batches(o, precision, batch_lo, batch_hi, st, [&](int64_t) -> int {
            cudaError_t e = tnk::launch_accumulate(root, E, uniq, P.k, R.n_sig, R.n_out, R.rank, amps, st);
            if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("accumulate: ") + cudaGetErrorString(e));
            return TN_OK;
        });
    };
    if (!P.opt.graphs || o->profile) {
        if (int rc = enqueue()) return rc;
        g_err.clear();
        return TN_OK;
    }
    const PlanObj::GraphKey key{precision, batch_lo, batch_hi, amps};
    auto it = o->graphs.find(key);
    if (it == o->graphs.end()) {
        // capture on a private stream (the caller's may be the legacy default
        // stream, which cannot be captured); nothing runs during capture
        if (!o->cap_stream) CU(cudaStreamCreateWithFlags(&o->cap_stream, cudaStreamNonBlocking));
        cudaGraph_t g = nullptr;
        cudaStream_t user = st;
        st = o->cap_stream;
        CU(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
        const int rc = enqueue();
        const cudaError_t ec = cudaStreamEndCapture(st, &g);
        st = user;
        if (rc) {
            if (g) cudaGraphDestroy(g);
            return rc;
        }
        if (ec != cudaSuccess) return set_err(TN_ECUDA, std::string("cudaStreamEndCapture: ") + cudaGetErrorString(ec));
        cudaGraphExec_t ex = nullptr;
        const cudaError_t ei = cudaGraphInstantiate(&ex, g, 0);
        cudaGraphDestroy(g);
        if (ei != cudaSuccess) return set_err(TN_ECUDA, std::string("cudaGraphInstantiate: ") + cudaGetErrorString(ei));
        it = o->graphs.emplace(key, ex).first;
    }
    CU(cudaGraphLaunch(it->second, st));
    g_err.clear();
    return TN_OK;
}

int tn_contract_slices(tn_plan_t plan, int precision, const int64_t *slice_ids, int32_t ns, double *partials,
                       void *stream) {
    if (!plan) return set_err(TN_EINVAL, "tn_contract_slices: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (!o->ws) return set_err(TN_ESTATE, "tn_contract_slices: no workspace bound");
    if (precision < TN_FP32 || precision > TN_BF16X3) return set_err(TN_EINVAL, "bad precision");
    if (ns < 0 || (ns > 0 && (!slice_ids || !partials))) return set_err(TN_EINVAL, "tn_contract_slices: bad args");
    tnp::Plan &P = o->P;
    const int64_t n_slices = int64_t(1) << P.sliced.size();
    const int64_t per = int64_t(1) << P.m_low;
    std::map<int64_t, std::vector<int32_t>> by_batch;
    std::vector<int64_t> internal(ns);
    for (int32_t i = 0; i < ns; ++i) {
        if (slice_ids[i] < 0 || slice_ids[i] >= n_slices) return set_err(TN_EINVAL, "slice id out of range");
        int64_t v = 0;  // external bit j = P.perm[t]  ->  internal bit t
        for (size_t t = 0; t < P.perm.size(); ++t) v |= ((slice_ids[i] >> P.perm[t]) & 1) << t;
        internal[i] = v;
        by_batch[v / per].push_back(i);
    }
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    const tnp::Node &R = P.nodes[P.root];
    const float2 *root = at<const float2>(o, R.buf.data);
    const int32_t *E = at<const int32_t>(o, R.buf.E);
    const int32_t *uniq = at<const int32_t>(o, P.off_uniq);
    // A pass computes the 2^m_low slices of a batch side by side; a pass per
    // slice computes just the instances of that slice (a step's time goes with
    // its instances: 16 slices of grid6x7_m10, 8 to a pass, took 19 ms each as
    // whole passes, 1.8 alone), but where launches and merged steps set the
    // time it is as long as a whole one.  Steps that no value of a sliced edge
    // changed for since the last pass keep their results: pass p re-runs the
    // levels up to the highest of a node that depends on a changed one.
    start_launches(o);
    struct Pos {
        int64_t b = -1, sigma = -1;  // batch, and slice of it (-1: a whole pass)
    } at_pos;
    auto level = [&](const Pos &prev, const Pos &next) -> int {
        if (prev.b < 0) return 64;
        int lv = next.b == prev.b ? -1 : 63 - __builtin_clzll((unsigned long long)(next.b ^ prev.b));
        for (const tnp::Node &nd : P.nodes) {
            if (nd.slices_low.empty()) continue;
            const bool same = next.sigma < 0 ? prev.sigma < 0
                                             : prev.sigma >= 0 && slice_instance(nd, next.sigma) ==
                                                                      slice_instance(nd, prev.sigma);
            if (!same) lv = std::max(lv, nd.level);
        }
        return lv;
    };
    std::map<std::pair<int, bool>, double> us;  // of a pass, by level and width
    auto estimate = [&](int lv, bool narrow) {
        auto it = us.find({lv, narrow});
        if (it == us.end()) it = us.emplace(std::make_pair(lv, narrow), pass_us(o, precision, lv, narrow)).first;
        return it->second;
    };
    auto pass = [&](int64_t b, int64_t sigma) -> int {
        const Pos next{b, sigma};
        const int lv = level(at_pos, next);
        at_pos = next;
        return lv >= 0 ? run_pass(o, precision, b, lv, sigma, st) : TN_OK;
    };
    auto extract = [&](int32_t i) -> int {
        cudaError_t e = tnk::launch_extract(root, E, uniq, P.k, internal[i] % per, R.n_out, R.rank,
                                            partials + (2 * P.k * i << R.rank), st);
        if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("extract: ") + cudaGetErrorString(e));
        return TN_OK;
    };
    for (auto &kv : by_batch) {
        std::map<int64_t, std::vector<int32_t>> by_slice;
        for (int32_t i : kv.second) by_slice[internal[i] % per].push_back(i);
        double narrow_us = 0.0;
        Pos p = at_pos;
        for (auto &ks : by_slice) {
            const Pos next{kv.first, ks.first};
            narrow_us += estimate(level(p, next), true);
            p = next;
        }
        const bool whole = narrow_us > estimate(level(at_pos, Pos{kv.first, -1}), false);
        if (whole)
            if (int rc = pass(kv.first, -1)) return rc;
        for (auto &ks : by_slice) {
            if (!whole)
                if (int rc = pass(kv.first, ks.first)) return rc;
            for (int32_t i : ks.second)
                if (int rc = extract(i)) return rc;
        }
    }
    o->last_batches = (int64_t)by_batch.size();
    g_err.clear();
    return TN_OK;
}

int tn_xeb(const double *amps, int64_t k, int32_t n_qubits, double *xeb_dev, void *stream) {
    if (!amps || !xeb_dev || k <= 0 || n_qubits < 1 || n_qubits > 1000)
        return set_err(TN_EINVAL, "tn_xeb: need k > 0, amplitudes and an output word");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = tnk::launch_xeb(amps, k, std::ldexp(1.0, n_qubits) / double(k), xeb_dev, st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("xeb: ") + cudaGetErrorString(e));
    g_err.clear();
    return TN_OK;
}

int tn_sample_completions(const double *amps, int64_t k, int32_t n_open, const double *uniform, int64_t *picks,
                          void *stream) {
    if (!amps || !uniform || !picks || k <= 0) return set_err(TN_EINVAL, "tn_sample_completions: need k > 0 and buffers");
    if (n_open < 0 || n_open > TN_MAX_OPEN) return set_err(TN_EINVAL, "tn_sample_completions: n_open outside [0, TN_MAX_OPEN]");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = tnk::launch_sample(amps, k, n_open, uniform, picks, st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("sample: ") + cudaGetErrorString(e));
    g_err.clear();
    return TN_OK;
}

int tn_pt_moments(const double *amps, int64_t k, int32_t n_qubits, double fidelity, double *out_dev, void *stream) {
    if (!amps || !out_dev || k <= 0 || n_qubits < 1 || n_qubits > 1000)
        return set_err(TN_EINVAL, "tn_pt_moments: need k > 0, amplitudes and 5 output words");
    if (!(fidelity >= 0.0 && fidelity < 1.0)) return set_err(TN_EINVAL, "tn_pt_moments: fidelity outside [0, 1)");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = tnk::launch_pt_moments(amps, k, std::ldexp(1.0, n_qubits), fidelity, out_dev, st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("pt_moments: ") + cudaGetErrorString(e));
    g_err.clear();
    return TN_OK;
}

size_t tn_pt_moments_scratch_bytes(int64_t k) { return k > 0 ? tnk::pt_moments_scratch_bytes(k) : 0; }

int tn_pt_moments_scratch(const double *amps, int64_t k, int32_t n_qubits, double fidelity, int32_t want_log,
                          double *out_dev, void *scratch, size_t scratch_bytes, void *stream) {
    if (!amps || !out_dev || !scratch || k <= 0 || n_qubits < 1 || n_qubits > 1000)
        return set_err(TN_EINVAL, "tn_pt_moments_scratch: need k > 0, amplitudes, 5 output words and scratch");
    if (!(fidelity >= 0.0 && fidelity < 1.0)) return set_err(TN_EINVAL, "tn_pt_moments_scratch: fidelity outside [0, 1)");
    if (scratch_bytes < tnk::pt_moments_scratch_bytes(k))
        return set_err(TN_ENOMEM, "tn_pt_moments_scratch: scratch needs " +
                                      std::to_string(tnk::pt_moments_scratch_bytes(k)) + " bytes");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = tnk::launch_pt_moments_scratch(amps, k, std::ldexp(1.0, n_qubits), fidelity, want_log != 0, out_dev,
                                                   static_cast<double *>(scratch), st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("pt_moments: ") + cudaGetErrorString(e));
    g_err.clear();
    return TN_OK;
}

int tn_pt_histogram(const double *amps, int64_t k, int32_t n_qubits, double x_max, int32_t nbins,
                    uint64_t *counts_dev, void *stream) {
    if (!amps || !counts_dev || k <= 0 || n_qubits < 1 || n_qubits > 1000)
        return set_err(TN_EINVAL, "tn_pt_histogram: need k > 0, amplitudes and a count array");
    if (nbins < 1 || nbins > TN_PT_MAX_BINS || !(x_max > 0.0))
        return set_err(TN_EINVAL, "tn_pt_histogram: need 1 <= nbins <= TN_PT_MAX_BINS and x_max > 0");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = tnk::launch_pt_hist(amps, k, std::ldexp(1.0, n_qubits), x_max, nbins,
                                        reinterpret_cast<unsigned long long *>(counts_dev), st);
    if (e != cudaSuccess) return set_err(TN_ECUDA, std::string("pt_histogram: ") + cudaGetErrorString(e));
    g_err.clear();
    return TN_OK;
}

int tn_plan_step_forms(tn_plan_t plan, int32_t *form, int32_t n) {
    if (!plan || (n > 0 && !form)) return set_err(TN_EINVAL, "tn_plan_step_forms: null argument");
    const PlanObj *o = reinterpret_cast<const PlanObj *>(plan);
    for (int32_t i = 0; i < n; ++i) form[i] = i < (int32_t)o->step_form.size() ? o->step_form[i] : -1;
    return TN_OK;
}

int tn_fma_probe(int64_t blocks, int64_t iters, float *out_dev, void *stream) {
    if (blocks <= 0 || blocks > 0x7fffffffLL || iters < 0 || !out_dev)
        return set_err(TN_EINVAL, "tn_fma_probe: need 0 < blocks < 2^31, iters >= 0 and an output buffer");
    CU(tnk::launch_fma_probe(blocks, iters, out_dev, reinterpret_cast<cudaStream_t>(stream)));
    g_err.clear();
    return TN_OK;
}

int tn_contract_static(tn_plan_t plan, int precision, double *amps, void *stream) {
    if (!plan) return set_err(TN_EINVAL, "tn_contract_static: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (o->P.ws_bytes > (int64_t)TN_STATIC_SCRATCH_BYTES)
        return set_err(TN_ENOMEM, "tn_contract_static: plan needs " + std::to_string(o->P.ws_bytes) +
                                      " workspace bytes; the fixed scratch holds " +
                                      std::to_string((long long)TN_STATIC_SCRATCH_BYTES));
    void *scratch = nullptr;
    if (int rc = static_scratch_address(&scratch)) return rc;
    // bind to the fixed scratch, run every batch, restore the caller's binding
    uint8_t *prev_ws = o->ws;
    const size_t prev_bytes = o->ws_bytes;
    int32_t *prev_flag = o->err_flag;
    const int32_t prev_graphs = o->P.opt.graphs;
    // graphs captured for the caller's own binding stay valid once it is
    // restored: keep them out of the re-bind's reach
    std::map<PlanObj::GraphKey, cudaGraphExec_t> kept;
    kept.swap(o->graphs);
    o->P.opt.graphs = 0;  // every call re-uploads the tables: nothing to replay
    int rc = tn_plan_bind(plan, scratch, (size_t)TN_STATIC_SCRATCH_BYTES, stream);
    if (rc == TN_OK) rc = tn_contract(plan, precision, 0, o->P.n_batches, amps, stream);
    if (rc == TN_OK) rc = tn_plan_check(plan, stream);
    const std::string msg = g_err;
    o->P.opt.graphs = prev_graphs;
    o->ws = prev_ws;
    o->ws_bytes = prev_bytes;
    o->err_flag = prev_flag;
    if (prev_ws) build_descs(o);
    else {
        o->desc.clear();
        o->amap.clear();
    }
    o->drop_graphs();  // none are captured while graphs are off; kept for symmetry
    o->graphs.swap(kept);
    g_err = msg;
    return rc;
}

int tn_plan_set_kernel(tn_plan_t plan, int32_t step, int32_t kernel) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_set_kernel: null plan");
    if (kernel < -1 || kernel > 1) return set_err(TN_EINVAL, "tn_plan_set_kernel: bad kernel family");
    return tn_plan_set_config(plan, step, kernel < 0 ? -1 : 2 * kernel);
}

int tn_plan_set_config(tn_plan_t plan, int32_t step, int32_t config) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_set_config: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    const tnp::Plan &P = o->P;
    if (step < 0 || step >= (int32_t)P.steps.size()) return set_err(TN_EINVAL, "tn_plan_set_config: bad step");
    const bool unfused = config >= TN_CONFIG_TUNED + TN_CONFIG_UNFUSED;
    if (unfused) config -= TN_CONFIG_UNFUSED;
    const bool tuned = config >= TN_CONFIG_TUNED;
    if (tuned) config -= TN_CONFIG_TUNED;
    if (config < -1 || config >= TN_NCONFIG) return set_err(TN_EINVAL, "tn_plan_set_config: bad configuration");
    if (config >= 0 && !config_allowed(P.steps[step], config))
        return set_err(TN_EINVAL, "tn_plan_set_config: per-row kernel needs N <= 16 and K*N <= 256");
    o->config_override.resize(P.steps.size(), -1);
    o->config_override[step] = config;
    // a step whose kernel was chosen runs by itself even if it is small
    o->pinned.resize(P.steps.size(), 0);
    o->pinned[step] = !tuned && config >= 0;
    // a chain that the plan formed by itself: run as its steps, or as the plan would
    const int c = P.steps[step].chain;
    if (!P.opt.fuse && c >= 0 && (unfused || config < 0)) {
        o->chain_on.resize(P.chains.size(), -1);
        o->chain_on[c] = unfused ? 0 : -1;
    }
    o->drop_graphs();
    return TN_OK;
}

int tn_plan_set_chain(tn_plan_t plan, int32_t chain, int32_t enable) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_set_chain: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (chain < 0 || chain >= o->reported_chains()) return set_err(TN_EINVAL, "tn_plan_set_chain: bad chain");
    o->chain_on.resize(o->P.chains.size(), -1);
    o->chain_on[chain] = enable ? 1 : 0;
    o->drop_graphs();
    return TN_OK;
}

int tn_plan_get_chains(tn_plan_t plan, int32_t *enabled, int32_t n) {
    if (!plan || (n > 0 && !enabled)) return set_err(TN_EINVAL, "tn_plan_get_chains: null argument");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    for (int32_t c = 0; c < n && c < o->reported_chains(); ++c) enabled[c] = o->chain_enabled(c) ? 1 : 0;
    return TN_OK;
}

int tn_plan_set_tc_resident_b(tn_plan_t plan, int32_t enable) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_set_tc_resident_b: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    o->tc_resident_b = enable != 0;
    o->drop_graphs();
    return TN_OK;
}

int tn_plan_set_tc_fp32(tn_plan_t plan, int32_t enable) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_set_tc_fp32: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    o->tc_fp32 = enable != 0;
    o->drop_graphs();
    return TN_OK;
}

int tn_plan_set_tc_pairs(tn_plan_t plan, int32_t enable) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_set_tc_pairs: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    o->tc_pair = enable != 0;
    o->drop_graphs();
    return TN_OK;
}

int tn_plan_get_configs(tn_plan_t plan, int32_t *config, int32_t n) {
    if (!plan || (n > 0 && !config)) return set_err(TN_EINVAL, "tn_plan_get_configs: null argument");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    for (int32_t s = 0; s < n && s < (int32_t)o->P.steps.size(); ++s) config[s] = effective_config(o, s);
    return TN_OK;
}

int tn_plan_get_choices(tn_plan_t plan, int32_t *choice, int32_t n) {
    if (!plan || (n > 0 && !choice)) return set_err(TN_EINVAL, "tn_plan_get_choices: null argument");
    const PlanObj *o = reinterpret_cast<const PlanObj *>(plan);
    for (int32_t s = 0; s < n && s < (int32_t)o->P.steps.size(); ++s) {
        const int32_t c = s < (int32_t)o->config_override.size() ? o->config_override[s] : -1;
        const bool pin = s < (int32_t)o->pinned.size() && o->pinned[s];
        const int ch = o->P.steps[s].chain;
        choice[s] = c;
        if (c >= 0 && !pin)
            choice[s] += TN_CONFIG_TUNED + (!o->P.opt.fuse && ch >= 0 && o->chain_state(ch) == 0 ? TN_CONFIG_UNFUSED : 0);
    }
    return TN_OK;
}

int tn_plan_features(tn_plan_t plan, int precision, int32_t config, float *feat, int32_t *eligible, int32_t n) {
    if (!plan || (n > 0 && !feat)) return set_err(TN_EINVAL, "tn_plan_features: null argument");
    if (precision < TN_FP32 || precision > TN_BF16X3) return set_err(TN_EINVAL, "tn_plan_features: bad precision");
    if (config < 0 || config >= TN_NCONFIG) return set_err(TN_EINVAL, "tn_plan_features: bad configuration");
    const PlanObj *o = reinterpret_cast<const PlanObj *>(plan);
    const tnp::Plan &P = o->P;
    for (int32_t s = 0; s < n && s < (int32_t)P.steps.size(); ++s) {
        step_features(o, s, precision, config, feat + int64_t(s) * TN_NFEAT);
        if (eligible) eligible[s] = config_allowed(P.steps[s], config) ? 1 : 0;
    }
    return TN_OK;
}

int tn_plan_autotune(tn_plan_t plan, int precision, int32_t reps, const uint8_t *step_mask, double *amps_scratch,
                     double *times, void *stream) {
    if (!plan || !amps_scratch) return set_err(TN_EINVAL, "tn_plan_autotune: null argument");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (!o->ws) return set_err(TN_ESTATE, "tn_plan_autotune: no workspace bound");
    if (precision < TN_FP32 || precision > TN_BF16X3) return set_err(TN_EINVAL, "tn_plan_autotune: bad precision");
    if (reps < 1) return set_err(TN_EINVAL, "tn_plan_autotune: reps must be >= 1");
    const tnp::Plan &P = o->P;
    const int ns = (int)P.steps.size();
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    // the steps' choices as they are (-1: the plan's own, which its rules may
    // take further than a configuration says)
    o->config_override.resize(ns, -1);
    const std::vector<int32_t> cur = o->config_override;
    std::vector<double> best(size_t(ns) * TN_NCONFIG, NAN), ms(ns);
    const bool prof = o->profile;
    o->profile = true;  // CUDA events around every step launch
    // Every step in a launch of its own; with a mask, the steps that are not
    // timed share launches as ever.
    // (A timed step runs the kernel that it will run by itself later.)
    if (step_mask) o->apart.assign(step_mask, step_mask + ns);
    else o->merge_small = false;
    o->config_override.assign(ns, -1);
    const int nchains = (int)P.chains.size();
    const std::vector<int8_t> prev_chain = o->chain_on;
    // configurations are timed on the separate steps; chains that hold no
    // selected step run as they would
    if (step_mask) {
        o->chain_on.resize(nchains, -1);
        for (int s = 0; s < ns; ++s)
            if (step_mask[s] && P.steps[s].chain >= 0) o->chain_on[P.steps[s].chain] = 0;
    } else {
        o->chain_on.assign(nchains, 0);
    }
    o->drop_graphs();
    int rc = TN_OK;
    for (int c = 0; c < TN_NCONFIG && rc == TN_OK; ++c) {
        bool any = false;
        for (int s = 0; s < ns; ++s) {
            const bool sel = (!step_mask || step_mask[s]) && config_allowed(P.steps[s], c);
            o->config_override[s] = sel ? c : cur[s];
            any = any || sel;
        }
        if (!any) continue;
        for (int r = 0; r <= reps && rc == TN_OK; ++r) {
            // the first slice batch of a call runs every step exactly once
            rc = tn_contract(plan, precision, 0, P.n_batches > 0 ? 1 : 0, amps_scratch, stream);
            if (rc == TN_OK) rc = tn_plan_step_times(plan, ms.data(), nullptr, ns);
            if (rc != TN_OK || r == 0) continue;  // the first run warms up
            for (int s = 0; s < ns; ++s) {
                if (o->config_override[s] != c || (step_mask && !step_mask[s])) continue;
                const double t = ms[s];
                double &b = best[size_t(s) * TN_NCONFIG + c];
                if (std::isnan(b) || t < b) b = t;
            }
        }
    }
    if (rc == TN_OK) rc = tn_plan_check(plan, stream);
    o->profile = prof;
    std::string msg = g_err;
    for (int s = 0; s < ns; ++s) {
        int pick = cur[s];
        if (rc == TN_OK && (!step_mask || step_mask[s])) {
            double bt = NAN;
            for (int c = 0; c < TN_NCONFIG; ++c) {
                const double t = best[size_t(s) * TN_NCONFIG + c];
                if (!std::isnan(t) && (std::isnan(bt) || t < bt)) {
                    bt = t;
                    pick = c;
                }
            }
        }
        o->config_override[s] = pick;
    }
    o->merge_small = true;
    o->apart.clear();
    // fused chains: each kept fused only where its kernel beats the sum of
    // its steps' best times (the chain's time is booked on its last step)
    // (with a step mask only some steps were timed: the chains keep their
    // previous setting)
    if (rc != TN_OK || step_mask) o->chain_on = prev_chain;
    o->drop_graphs();
    if (rc == TN_OK && nchains > 0 && !step_mask) {
        std::vector<double> unfused(nchains, 0.0), fused(nchains, NAN);
        for (int s = 0; s < ns; ++s) {
            const int c = P.steps[s].chain;
            if (c < 0) continue;
            double bt = NAN;
            for (int k = 0; k < TN_NCONFIG; ++k) {
                const double t = best[size_t(s) * TN_NCONFIG + k];
                if (!std::isnan(t) && (std::isnan(bt) || t < bt)) bt = t;
            }
            unfused[c] += std::isnan(bt) ? 0.0 : bt;
        }
        for (int c = 0; c < nchains; ++c) o->chain_on[c] = o->chain_small[c] ? 0 : 1;
        o->drop_graphs();
        o->profile = true;
        for (int r = 0; r <= reps && rc == TN_OK; ++r) {
            rc = tn_contract(plan, precision, 0, P.n_batches > 0 ? 1 : 0, amps_scratch, stream);
            if (rc == TN_OK) rc = tn_plan_step_times(plan, ms.data(), nullptr, ns);
            if (rc != TN_OK || r == 0) continue;
            for (int s = 0; s < ns; ++s) {
                const tnp::Step &S = P.steps[s];
                if (S.chain < 0 || !S.chain_last) continue;
                if (std::isnan(fused[S.chain]) || ms[s] < fused[S.chain]) fused[S.chain] = ms[s];
            }
        }
        if (rc == TN_OK) rc = tn_plan_check(plan, stream);
        if (rc != TN_OK) msg = g_err;
        o->profile = prof;
        for (int c = 0; c < nchains; ++c) o->chain_on[c] = (!std::isnan(fused[c]) && fused[c] < unfused[c]) ? 1 : 0;
        if (rc != TN_OK) o->chain_on = prev_chain;
        // (chains of small steps only stay among the plan's other small steps
        // in their merged launches: a phase there costs a tenth of a kernel)
        for (int c = 0; c < nchains; ++c)
            if (rc == TN_OK && o->chain_small[c]) o->chain_on[c] = 0;
    }
    o->drop_graphs();
    if (times) std::copy(best.begin(), best.end(), times);
    g_err = rc == TN_OK ? std::string() : msg;
    return rc;
}

int tn_plan_select(tn_plan_t plan, int precision, const uint16_t *params16, float margin, void *scratch,
                   size_t scratch_bytes, int32_t *uncertain, void *stream) {
    if (!plan || !params16 || !scratch) return set_err(TN_EINVAL, "tn_plan_select: null argument");
    if (precision < TN_FP32 || precision > TN_BF16X3) return set_err(TN_EINVAL, "tn_plan_select: bad precision");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    const tnp::Plan &P = o->P;
    const int ns = (int)P.steps.size();
    const int64_t rows = int64_t(ns) * TN_NCONFIG;
    const size_t need = size_t(rows) * (TN_NFEAT + 1) * sizeof(float);
    if (scratch_bytes < need)
        return set_err(TN_ENOMEM, "tn_plan_select: scratch needs " + std::to_string(need) + " bytes");
    std::vector<float> X(size_t(rows) * TN_NFEAT), y(rows);
    for (int s = 0; s < ns; ++s)
        for (int c = 0; c < TN_NCONFIG; ++c) step_features(o, s, precision, c, &X[(size_t(s) * TN_NCONFIG + c) * TN_NFEAT]);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    float *dX = static_cast<float *>(scratch), *dy = dX + rows * TN_NFEAT;
    CU(cudaMemcpyAsync(dX, X.data(), X.size() * sizeof(float), cudaMemcpyHostToDevice, st));
    CU(tnk::mlp_forward_f16(params16, dX, rows, dy, st));
    CU(cudaMemcpyAsync(y.data(), dy, y.size() * sizeof(float), cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    o->config_override.resize(ns, -1);
    for (int s = 0; s < ns; ++s) {
        int b1 = -1;
        float y1 = 0.f, y2 = 0.f;
        bool have2 = false;
        tnk::StepDesc t = shape_desc(o, P.steps[s]);
        // FMAs (3) are at most 5 % faster where BF16x6 (2) applies (one of 70
        // measured steps; the median takes 3.1 times as long), and its rows
        // are rare in a corpus: not left to the network
        const bool split = precision == TN_FP32 && step_form(t, 2, false, precision, 1, true) == TN_FORM_TC_FP32;
        for (int c = 0; c < TN_NCONFIG; ++c) {
            if (!config_allowed(P.steps[s], c) || (split && c == 3)) continue;
            const float v = y[size_t(s) * TN_NCONFIG + c];
            if (b1 < 0 || v < y1) {
                if (b1 >= 0) {
                    y2 = y1;
                    have2 = true;
                }
                y1 = v;
                b1 = c;
            } else if (!have2 || v < y2) {
                y2 = v;
                have2 = true;
            }
        }
        o->config_override[s] = b1;
        // (a small step that shares a launch, one of a fused chain and one of few
        // multiply-adds run the same whatever is chosen)
        const bool same = merges(o, s) || o->chain_fused(P.steps[s].chain) ||
                          tnk::step_few_takes(shape_desc(o, P.steps[s]), precision != TN_FP32, false);
        if (uncertain) uncertain[s] = (have2 && y2 - y1 < margin && !same) ? 1 : 0;
    }
    o->drop_graphs();
    g_err.clear();
    return TN_OK;
}

size_t tn_mlp_grad_scratch_bytes(int64_t n) { return tnk::mlp_grad_scratch_bytes(n); }

int tn_mlp_forward(const float *params, const float *X, int64_t n, float *y, void *stream) {
    if (!params || n < 0 || (n > 0 && (!X || !y))) return set_err(TN_EINVAL, "tn_mlp_forward: bad arguments");
    CU(tnk::mlp_forward(params, X, n, y, reinterpret_cast<cudaStream_t>(stream)));
    return TN_OK;
}

int tn_mlp_grad(const float *params, const float *X, const float *t, int64_t n, float *grad, float *loss,
                void *scratch, size_t scratch_bytes, void *stream) {
    if (!params || !X || !t || !grad || !scratch || n <= 0) return set_err(TN_EINVAL, "tn_mlp_grad: bad arguments");
    if (scratch_bytes < tnk::mlp_grad_scratch_bytes(n))
        return set_err(TN_ENOMEM, "tn_mlp_grad: scratch needs " + std::to_string(tnk::mlp_grad_scratch_bytes(n)) +
                                      " bytes");
    CU(tnk::mlp_grad(params, X, t, n, grad, loss, static_cast<float *>(scratch), reinterpret_cast<cudaStream_t>(stream)));
    return TN_OK;
}

int tn_mlp_adam(float *params, const float *grad, float *m, float *v, int32_t step, float lr, float beta1,
                float beta2, float eps, void *stream) {
    if (!params || !grad || !m || !v || step < 1) return set_err(TN_EINVAL, "tn_mlp_adam: bad arguments");
    CU(tnk::mlp_adam(params, grad, m, v, step, lr, beta1, beta2, eps, reinterpret_cast<cudaStream_t>(stream)));
    return TN_OK;
}

int tn_mlp_to_half(const float *params, uint16_t *params16, void *stream) {
    if (!params || !params16) return set_err(TN_EINVAL, "tn_mlp_to_half: null argument");
    CU(tnk::mlp_to_half(params, params16, reinterpret_cast<cudaStream_t>(stream)));
    return TN_OK;
}

int tn_mlp_forward_f16(const uint16_t *params16, const float *X, int64_t n, float *y, void *stream) {
    if (!params16 || n < 0 || (n > 0 && (!X || !y))) return set_err(TN_EINVAL, "tn_mlp_forward_f16: bad arguments");
    CU(tnk::mlp_forward_f16(params16, X, n, y, reinterpret_cast<cudaStream_t>(stream)));
    return TN_OK;
}

int tn_plan_check(tn_plan_t plan, void *stream) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_check: null plan");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    if (!o->ws) return TN_OK;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    int32_t flag = 0;
    CU(cudaMemcpyAsync(&flag, o->err_flag, 4, cudaMemcpyDeviceToHost, st));
    CU(cudaStreamSynchronize(st));
    if (flag) {
        CU(cudaMemsetAsync(o->err_flag, 0, 4, st));
        CU(cudaStreamSynchronize(st));
        return set_err(TN_ETIMEOUT, "a bounded device-side wait gave up (tensor-core pipeline)");
    }
    return TN_OK;
}

int tn_plan_profile(tn_plan_t plan, int enable) {
    if (!plan) return set_err(TN_EINVAL, "tn_plan_profile: null plan");
    reinterpret_cast<PlanObj *>(plan)->profile = enable != 0;
    return TN_OK;
}

int tn_plan_step_times(tn_plan_t plan, double *ms, int32_t *kernel, int32_t n) {
    if (!plan || !ms) return set_err(TN_EINVAL, "tn_plan_step_times: null argument");
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    for (int32_t i = 0; i < n; ++i) {
        ms[i] = 0.0;
        if (kernel) kernel[i] = i < (int32_t)o->step_kernel.size() ? o->step_kernel[i] : -1;
    }
    for (size_t q = 0; q < o->ev_used; ++q) {
        CU(cudaEventSynchronize(o->ev[2 * q + 1]));
        float t = 0.f;
        CU(cudaEventElapsedTime(&t, o->ev[2 * q], o->ev[2 * q + 1]));
        if (o->ev_step[q] < n) ms[o->ev_step[q]] += t;
    }
    return TN_OK;
}

void tn_destroy(tn_plan_t plan) {
    if (!plan) return;
    PlanObj *o = reinterpret_cast<PlanObj *>(plan);
    o->drop_graphs();
    if (o->cap_stream) cudaStreamDestroy(o->cap_stream);
    for (cudaEvent_t e : o->ev) cudaEventDestroy(e);
    delete o;
}

}  // extern "C"
