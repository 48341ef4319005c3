"""The work that users of this framework have it do, as cases to be timed.

Kinds of case (the ``kind`` field):

* ``amplitudes``: amplitudes of a batch of bitstrings, every slice batch of a
  bound plan (``Plan.tn_contract``); with ``open`` > 0 correlated batches and
  one perfect sample per row (``tn_sample_completions``) behind them.
* ``slices``: partial amplitudes of individual slices
  (``Plan.tn_contract_slices``).
* ``stream``: successive bitstring batches from host arrays to host arrays
  (``pipeline.contract_batches``): planning, table upload, contraction and
  read-back, overlapped.
* ``sample``: perfect samples from correlated batches held on the device.
* ``fidelity``: linear XEB, Porter-Thomas fit and histogram of a set of
  amplitudes (``tn_xeb``, ``xeb.porter_thomas_fit``, ``porter_thomas_histogram``).
* ``mlp_train``: one training step of the cost model (``tn_mlp_grad``,
  ``tn_mlp_adam``); ``mlp_predict``: its FP16 inference over a corpus.

``exact`` evaluates the same in 64 bits with plain torch / numpy: circuits of
up to 30 qubits by a state vector, larger ones by a pairwise contraction of
the unfused bookkeeping below for a few of the rows.
"""

import functools
import math

import numpy as np
import torch

from paper_2212_04749_gb300 import tn, xeb
from paper_2212_04749_gb300.pipeline import contract_batches
from rqc import diamond_layout, grid_layout, make_workload, network_structure, random_circuit
from rqc.bitstrings import uniform_bitstrings
from rqc.tree import ContractionTree, candidate_trees, choose_slices, estimate_cost

GIB = 1 << 30
D, H = tn.TN_MLP_IN, tn.TN_MLP_HIDDEN
EXACT_ROWS = 32    # rows checked of a circuit too large for a state vector
EXACT_SLICES = 2   # slices checked of a sliced one


def listed():
    return [
        # one small circuit, few bitstrings: the call a user makes while trying things
        # out; launches and latency are all of it
        {"name": "amps_3x4_fp32", "kind": "amplitudes", "workload": "grid3x4_m8", "rows": 64, "prec": "fp32"},
        # a 20-qubit circuit, ragged row count, two sliced edges, the quick tensor form
        {"name": "amps_4x5_tf32", "kind": "amplitudes", "layout": "4x5", "cycles": 12, "circuit": 21, "rows": 1500,
         "slices": 2, "prec": "tf32"},
        # 30 qubits, 4096 bitstrings, 2^10 slices in 16 batches, default options
        {"name": "amps_5x6_bf16x3", "kind": "amplitudes", "workload": "grid5x6_m14", "rows": 4096,
         "prec": "bf16x3", "ws_gib": 24},
        # a rank's check of single slices of a heavily sliced 42-qubit circuit
        {"name": "slices_6x7_bf16x3", "kind": "slices", "workload": "grid6x7_m10", "trials": 2, "rows": 64,
         "n_ids": 16, "prec": "bf16x3", "ws_gib": 24},
        # the headline workload: 53 qubits, 8192 bitstrings, tuned plan, chains fused where faster
        {"name": "amps_diamond53_bf16x3", "kind": "amplitudes", "workload": "diamond53_m12", "rows": 8192,
         "prec": "bf16x3", "tuned": True, "fuse": 1, "ws_gib": 40},
        # the same in plain FP32, the reference form that the mixed ones are held against
        {"name": "amps_diamond53_fp32", "kind": "amplitudes", "workload": "diamond53_m12", "rows": 8192,
         "prec": "fp32", "tuned": True, "fuse": 1, "ws_gib": 40},
        # correlated batches: 256 rows with 4 open qubits, then one perfect sample per row
        {"name": "correlated_diamond53", "kind": "amplitudes", "workload": "diamond53_m12", "rows": 256, "open": 4,
         "prec": "bf16x3", "ws_gib": 40},
        # many perfect samples from stored correlated batches
        {"name": "sample_8192x1024", "kind": "sample", "rows": 8192, "open": 10},
        # the fidelity of a three-million-amplitude run
        {"name": "fidelity_3m", "kind": "fidelity", "rows": 3000000, "qubits": 53, "bins": 64},
        # one optimiser step of the cost model at its training batch
        {"name": "mlp_train_4096", "kind": "mlp_train", "rows": 4096},
        # the cost model over a corpus of (step, configuration) rows
        {"name": "mlp_predict_104622", "kind": "mlp_predict", "rows": 104622},
        # a service answering batch after batch of 20-qubit requests
        {"name": "stream_4x5_bf16x3", "kind": "stream", "layout": "4x5", "cycles": 12, "circuit": 21, "rows": 1500,
         "slices": 0, "batches": 6, "prec": "bf16x3"},
    ]


def _log(rng, lo, hi):
    """A whole number of [lo, hi], spread over the logarithm, odd ones as likely as even ones."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def _draw_circuit(rng, case, flops, peak):
    """Adds a circuit to a case whose contraction stays below `flops` and `peak` bytes per tensor."""
    while True:
        r, c = rng.randint(3, 5), rng.randint(3, 6)
        if r * c > 30:
            continue
        case.update(layout="%dx%d" % (r, c), cycles=rng.randint(5, 14), circuit=rng.randrange(1 << 30),
                    slices=rng.choice((0, 0, 0, 1, 2, 3, 5)))
        if case.get("open"):
            case["slices"] = 0
        _, _, struct, ssa, sliced = _network(_key(case))
        cost = estimate_cost(struct, ssa, case["rows"], sliced)
        grow = 1 << case.get("open", 0)
        if cost.flops * grow * case.get("batches", 1) <= flops and cost.peak_bytes * grow <= peak:
            return case


def draw(rng):
    kind = rng.choice(("amplitudes",) * 6 + ("slices", "stream", "sample", "fidelity", "mlp_train", "mlp_predict"))
    case = {"kind": kind}
    if kind in ("amplitudes", "slices", "stream"):
        case["prec"] = rng.choice(("fp32", "tf32", "bf16x3", "bf16x3"))
        case["rows"] = _log(rng, 1, 8192)
    if kind == "amplitudes":
        case["fuse"] = rng.choice((0, 0, 1))
        if rng.random() < 0.25:
            case["open"] = rng.randint(1, 6)
            case["rows"] = _log(rng, 1, 512)
        elif rng.random() < 0.2:  # the 53-qubit circuit along its stored tree
            case.update(workload="diamond53_m12", rows=_log(rng, 16, 8192), ws_gib=40)
            return case
        return _draw_circuit(rng, case, 4e12, 4 * GIB)
    if kind == "slices":
        case["n_ids"] = rng.randint(1, 4)
        case = _draw_circuit(rng, case, 1e12, 2 * GIB)
        if case["slices"] < 2:
            case["slices"] = 2
        return case
    if kind == "stream":
        case.update(batches=rng.randint(1, 8), rows=_log(rng, 1, 4096))
        return _draw_circuit(rng, case, 1e11, GIB // 4)
    if kind == "sample":
        case["open"] = rng.randint(0, 16)
        case["rows"] = _log(rng, 1, max(1, min(65536, (1 << 23) >> case["open"])))
    elif kind == "fidelity":
        case.update(rows=_log(rng, 64, 3000000), qubits=rng.randint(12, 60), bins=_log(rng, 8, 1024))
    elif kind == "mlp_train":
        case["rows"] = _log(rng, 64, 16384)
    else:
        case["rows"] = _log(rng, 64, 131072)
    return case


def _key(case):
    return (case.get("workload", ""), case.get("trials", 1), case.get("layout", ""), case.get("cycles", 0),
            case.get("circuit", 0), case.get("slices", 0), case["rows"])


@functools.lru_cache(maxsize=16)
def _network(key):
    """(circuit, its C form's arrays kept by it, structure, tree, sliced edges) of a case."""
    workload, trials, layout, cycles, seed, slices, rows = key
    if workload:
        # the stored tree where the workload has one, else the seeded search
        stored = workload.startswith("diamond53")
        w = make_workload(workload) if stored else make_workload(workload, trials=trials)
        return w.circuit, w.name, w.struct, w.tree.ssa, list(w.tree.sliced)
    r, c = (int(x) for x in layout.split("x"))
    circ = random_circuit(grid_layout(r, c), cycles, seed=seed)
    struct = network_structure(circ)
    ssa = candidate_trees(struct, rows, seed=2, trials=1)[0]
    sliced = choose_slices(struct, ContractionTree(ssa=ssa), rows, n_sliced=slices) if slices else []
    return circ, layout, struct, ssa, sliced


def _options(case):
    o = {"workspace_limit": case.get("ws_gib", 16) * GIB}
    if case.get("fuse"):
        o.update(fuse=1, fuse_max_bits=9)
    return o


def _open_qubits(n, r):
    return list(range(n - r, n))


def _bits(case, n, seed, batch=0):
    return uniform_bitstrings(n, case["rows"], seed=(int(seed) << 8) + batch)


def _slice_ids(case, seed, n_sliced):
    return np.random.default_rng([int(seed), 7]).choice(1 << n_sliced, case["n_ids"], replace=False).astype(np.int64)


def _batch_amplitudes(case, seed):
    """rows x 2^open complex amplitudes of correlated batches: Gaussian, as deep random circuits give them."""
    g = torch.Generator().manual_seed(int(seed))
    return torch.randn(case["rows"] << case["open"], 2, generator=g, dtype=torch.float64)


def _run_amplitudes(case, seed):
    """complex amplitudes of `rows` samples of fidelity 0.3: |amp|^2 2^n from x e^-x with weight 0.3, else e^-x."""
    g = torch.Generator().manual_seed(int(seed))
    k = case["rows"]
    u, v, pick, arg = torch.rand(4, k, generator=g, dtype=torch.float64)
    x = -torch.log1p(-u) - torch.where(pick < 0.3, torch.log1p(-v), torch.zeros(k, dtype=torch.float64))
    r = torch.sqrt(x) * 2.0 ** (-0.5 * case["qubits"])
    return torch.stack([r * torch.cos(2 * math.pi * arg), r * torch.sin(2 * math.pi * arg)], 1).contiguous()


def _mlp_inputs(case, seed):
    """A cost-model network in mid-training (moments in place), step features in [0, 1] and log2 times."""
    g = torch.Generator().manual_seed(int(seed))

    def uniform(*shape):
        return torch.rand(*shape, generator=g) * 2 - 1

    p = torch.cat([uniform(H * D) * math.sqrt(6 / D), 0.1 * uniform(H), uniform(H * H) * math.sqrt(6 / H),
                   0.1 * uniform(H), uniform(H) * math.sqrt(3 / H), uniform(1)])
    n = case["rows"]
    X = torch.rand(n, D, generator=g)
    t = torch.sin(3 * X[:, 0]) + X[:, 1] * X[:, 2] - 4
    m = 1e-3 * torch.randn(p.numel(), generator=g)
    v = 1e-5 * (0.5 + torch.rand(p.numel(), generator=g))
    return p, X, t, m, v


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "stream": torch.cuda.current_stream()}
    if kind in ("amplitudes", "slices"):
        circ, _, _, ssa, sliced = _network(_key(case))
        n, r = circ.n_qubits, case.get("open", 0)
        opts = _options(case)
        if r:
            opts["open_qubits"] = _open_qubits(n, r)
        plan = tn.Plan(circ, _bits(case, n, seed), ssa, sliced, **opts)
        s["plan"] = plan
        s["ws"] = torch.empty(max(plan.info["workspace_bytes"], 256), dtype=torch.uint8, device="cuda")
        plan.tn_plan_bind(s["ws"], stream=s["stream"])
        if kind == "slices":
            s["ids"] = _slice_ids(case, seed, len(sliced))
            s["out"] = torch.zeros(case["n_ids"], case["rows"], 2, dtype=torch.float64, device="cuda")
            return s
        s["amps"] = torch.zeros(case["rows"], 1 << r, 2, dtype=torch.float64, device="cuda")
        if r:
            s["u"] = torch.from_numpy(np.random.default_rng(int(seed)).random(case["rows"])).cuda()
            s["picks"] = torch.zeros(case["rows"], dtype=torch.int64, device="cuda")
        if case.get("tuned"):
            plan.tn_plan_autotune(case["prec"], s["amps"], reps=2, stream=s["stream"])
    elif kind == "stream":
        circ, _, _, ssa, sliced = _network(_key(case))
        s["bits"] = [_bits(case, circ.n_qubits, seed, b) for b in range(case["batches"])]
        s["net"] = circ, ssa, sliced
        # room for any batch of this size (plans differ a little with the bitstrings)
        need = max(tn.Plan(circ, b, ssa, sliced, **_options(case)).info["workspace_bytes"] for b in s["bits"])
        s["ws"] = [torch.empty(max(need, 256), dtype=torch.uint8, device="cuda") for _ in range(3)]
    elif kind == "sample":
        s["amps"] = _batch_amplitudes(case, seed).cuda()
        s["u"] = torch.from_numpy(np.random.default_rng(int(seed)).random(case["rows"])).cuda()
        s["picks"] = torch.zeros(case["rows"], dtype=torch.int64, device="cuda")
    elif kind == "fidelity":
        s["amps"] = _run_amplitudes(case, seed).cuda()
        s["xeb"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    else:
        p, X, t, m, v = (x.cuda() for x in _mlp_inputs(case, seed))
        s.update(X=X, t=t, p=p, m=m, v=v)
        if kind == "mlp_train":
            s["grad"], s["loss"] = torch.zeros_like(p), torch.zeros(1, device="cuda")
            s["scratch"] = torch.empty(tn.tn_mlp_grad_scratch_bytes(case["rows"]), dtype=torch.uint8, device="cuda")
            s["step"] = 200
        else:
            s["p16"] = torch.zeros(p.numel(), dtype=torch.int16, device="cuda")
            tn.tn_mlp_to_half(p, s["p16"], stream=s["stream"])
            s["y"] = torch.zeros(case["rows"], device="cuda")
    return s


def run(s):
    case, st = s["case"], s["stream"]
    kind = case["kind"]
    if kind == "amplitudes":
        s["amps"].zero_()
        s["plan"].tn_contract(s["amps"], case["prec"], stream=st)
        if not case.get("open"):
            return _split(s["amps"], case, EXACT_ROWS)
        tn.tn_sample_completions(s["amps"], case["rows"], case["open"], s["u"], s["picks"], stream=st)
        return _split(s["amps"], case, EXACT_ROWS) + [s["picks"]]
    if kind == "slices":
        s["plan"].tn_contract_slices(s["ids"], s["out"], case["prec"], stream=st)
        return _split(s["out"], case, EXACT_SLICES)
    if kind == "stream":
        circ, ssa, sliced = s["net"]
        return [a for _, a in contract_batches(circ, s["bits"], ssa, sliced, case["prec"], s["ws"], stream=st,
                                               **_options(case))]
    if kind == "sample":
        tn.tn_sample_completions(s["amps"], case["rows"], case["open"], s["u"], s["picks"], stream=st)
        return s["picks"]
    if kind == "fidelity":
        k, n = case["rows"], case["qubits"]
        tn.tn_xeb(s["amps"], k, n, s["xeb"], stream=st)
        fit = xeb.porter_thomas_fit(s["amps"], k, n, stream=st)
        counts = xeb.porter_thomas_histogram(s["amps"], k, n, nbins=case["bins"], stream=st)
        return {"xeb": s["xeb"], "counts": counts,
                "fit": {f: fit[f] for f in ("fidelity", "stderr", "loglik", "linear", "linear_stderr")}}
    if kind == "mlp_train":
        s["step"] += 1
        tn.tn_mlp_grad(s["p"], s["X"], s["t"], case["rows"], s["grad"], s["loss"], s["scratch"], stream=st)
        tn.tn_mlp_adam(s["p"], s["grad"], s["m"], s["v"], s["step"], lr=2e-3, stream=st)
        return {"params": s["p"], "m": s["m"], "v": s["v"], "grad": s["grad"], "loss": s["loss"]}
    tn.tn_mlp_forward_f16(s["p16"], s["X"], case["rows"], s["y"], stream=st)
    return s["y"]


def _whole(case):
    """Whether exact() covers every row (state vector) or only the first ones."""
    if "layout" in case:
        return True
    return case["workload"] in ("grid3x4_m8", "grid5x6_m14")


def _split(out, case, head):
    """The output whole, in two parts where only the first of its rows has an exact value."""
    return [out] if _whole(case) and case["kind"] == "amplitudes" else [out[:head], out[head:]]


def work(case):
    kind, k = case["kind"], case["rows"]
    if kind in ("amplitudes", "slices", "stream"):
        circ, _, struct, ssa, sliced = _network(_key(case))
        n, r = circ.n_qubits, case.get("open", 0)
        flops = estimate_cost(struct, ssa, k, sliced).flops
        if r:  # open qubits raise the ranks of the tensors above them
            flops = tn.Plan(circ, _bits(case, n, 0), ssa, sliced, open_qubits=_open_qubits(n, r), **_options(case)).info["flops_ma"]
        outs, passes = k << r, case.get("batches", 1)
        if kind == "slices":
            passes, outs = case["n_ids"], k
            flops /= 1 << len(sliced)
        # the gates, the bitstrings, the amplitudes
        return {"bytes": 256 * struct.n_tensors + passes * (k * n + 16 * outs), "flops": flops * passes}
    if kind == "sample":
        return {"bytes": 16 * (k << case["open"]) + 16 * k, "flops": 4 * (k << case["open"])}
    if kind == "fidelity":
        return {"bytes": 16 * k + 8 * case["bins"], "flops": 40 * k}
    flops = 2 * (D * H + H * H + H) * k
    if kind == "mlp_train":
        return {"bytes": 4 * k * (D + 1) + 7 * 4 * tn.TN_MLP_NPARAMS, "flops": 3 * flops}
    return {"bytes": 4 * k * (D + 1) + 2 * tn.TN_MLP_NPARAMS, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    # about four times the error against 64 bits
    if kind == "sample":
        return "exact"  # ordered, correctly rounded FP64 sums and comparisons
    if kind == "fidelity":
        return {"rel": 1e-11}  # FP64 sums; the fit stops at steps of 1e-13
    if kind == "mlp_train":
        return {"rel": 2e-6}  # FP32 sums over the rows and 128 units: 3e-7
    if kind == "mlp_predict":
        return {"rel": 5e-3}  # FP16 weights and activations: 1.1e-3
    # FP32 1.4e-6, BF16x3 3.3e-5 on the 53-qubit circuit; TF32 2.3e-2 there, 5e-3 on the grids
    rel = {"fp32": 6e-6, "tf32": 2e-2 if "layout" in case else 8e-2, "bf16x3": 1.4e-4}[case["prec"]]
    if case.get("open"):
        return {"rel": rel, "differ": 0.05}  # a sample moves where its number lies at a border
    return {"rel": rel}


# ---------------------------------------------------------------- 64 bits

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _state(circ):
    """|psi> = U |0..0>, complex128, qubit 0 the most significant bit; single-qubit gates ride on the next
    two-qubit gate of their qubit, the last ones follow."""
    n, dev = circ.n_qubits, _device()
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=dev)
    psi[0] = 1
    wait = [np.eye(2, dtype=np.complex128) for _ in range(n)]
    for g in circ.gates:
        if len(g.qubits) == 1:
            wait[g.qubits[0]] = g.matrix @ wait[g.qubits[0]]
            continue
        a, b = g.qubits
        m = g.matrix @ np.kron(wait[a], wait[b])
        wait[a] = wait[b] = np.eye(2, dtype=np.complex128)
        m = torch.from_numpy(m).to(dev).reshape(2, 2, 2, 2)
        psi = psi.view(1 << a, 2, 1 << (b - a - 1), 2, 1 << (n - 1 - b))
        new = torch.empty_like(psi)
        for x in range(2):
            for y in range(2):
                part = new[:, x, :, y]
                part.copy_(psi[:, 0, :, 0]).mul_(m[x, y, 0, 0])
                for u, v in ((0, 1), (1, 0), (1, 1)):
                    part.addcmul_(psi[:, u, :, v], m[x, y, u, v])
        psi = new.view(-1)
    for q in range(n):
        psi = psi.view(1 << q, 2, -1)
        m = torch.from_numpy(wait[q]).to(dev)
        psi = torch.stack([m[0, 0] * psi[:, 0] + m[0, 1] * psi[:, 1], m[1, 0] * psi[:, 0] + m[1, 1] * psi[:, 1]], 1)
    return psi.reshape(-1)


def _real(z):
    return torch.view_as_real(z).contiguous()


def _index(bits):
    n = bits.shape[1]
    return torch.from_numpy((bits.astype(np.int64) << np.arange(n - 1, -1, -1)).sum(1))


def _tensors(circ):
    """One tensor per two-qubit gate, legs (out a, out b, in a, in b), with the bond edges (numbered as the wires
    between gates appear) and the output qubits on its legs; -1: no leg there (|0> put in)."""
    wait = {q: np.eye(2, dtype=np.complex128) for q in range(circ.n_qubits)}
    last, made, edges = {}, [], 0
    for g in circ.gates:
        if len(g.qubits) == 1:
            wait[g.qubits[0]] = g.matrix @ wait[g.qubits[0]]
            continue
        a, b = g.qubits
        t = (g.matrix @ np.kron(wait[a], wait[b])).reshape(2, 2, 2, 2)
        wait[a] = wait[b] = np.eye(2, dtype=np.complex128)
        legs = [None, None, None, None]
        for j, q in enumerate((a, b)):
            if q in last:
                made[last[q][0]][1][last[q][1]] = ("e", edges)
                legs[2 + j] = ("e", edges)
                edges += 1
        for j, q in enumerate((a, b)):
            last[q] = (len(made), j)
        made.append([t, legs])
    for q, (i, j) in last.items():
        made[i][0] = np.moveaxis(np.tensordot(wait[q], made[i][0], axes=(1, j)), 0, j)
        made[i][1][j] = ("q", q)
    return made


def _contract(circ, ssa, rows, fixed, open_qubits=()):
    """Amplitudes of bitstrings `rows` along a tree, each distinct projection of the rows once; `fixed`: bond edge ->
    value. A node: (edges of its tensor's axes after the first, instance of each row, tensor)."""
    dev = _device()
    nodes = []
    for t, legs in _tensors(circ):
        axes, cols, at = [], [], []
        for j, leg in enumerate(legs):
            if leg is None:
                t = np.take(t, [0], axis=j)
            elif leg[0] == "e" and leg[1] in fixed:
                t = np.take(t, [fixed[leg[1]]], axis=j)
            elif leg[0] == "e":
                axes.append((leg[1], j))
            elif leg[1] in open_qubits:
                axes.append(("q%d" % leg[1], j))
            else:
                cols.append(rows[:, leg[1]])
                at.append(j)
        order = at + [j for _, j in axes] + [j for j in range(4) if j not in at and j not in [x for _, x in axes]]
        t = torch.from_numpy(np.ascontiguousarray(t.transpose(order))).to(dev)
        t = t.reshape([1 << len(at)] + [2] * len(axes))
        inst = sum((c.astype(np.int64) << (len(cols) - 1 - i) for i, c in enumerate(cols)), np.zeros(len(rows), np.int64))
        nodes.append(([e for e, _ in axes], inst, t))
    for a, b in np.asarray(ssa):
        (ea, ia, ta), (eb, ib, tb) = nodes[a], nodes[b]
        nodes[a] = nodes[b] = None
        both = [e for e in ea if e in eb]
        ra, rb = [e for e in ea if e not in both], [e for e in eb if e not in both]
        pairs, inst = np.unique(np.stack([ia, ib], 1), axis=0, return_inverse=True)
        ta = ta.permute([0] + [1 + ea.index(e) for e in ra + both]).reshape(ta.shape[0], 1 << len(ra), 1 << len(both))
        tb = tb.permute([0] + [1 + eb.index(e) for e in both + rb]).reshape(tb.shape[0], 1 << len(both), 1 << len(rb))
        out = torch.empty(len(pairs), 1 << len(ra), 1 << len(rb), dtype=torch.complex128, device=dev)
        for i, (x, y) in enumerate(pairs):
            torch.matmul(ta[x], tb[y], out=out[i])
        nodes.append((ra + rb, inst.reshape(-1), out.reshape([len(pairs)] + [2] * (len(ra) + len(rb)))))
    e, inst, t = nodes[-1]
    t = t.permute([0] + [1 + e.index("q%d" % q) for q in open_qubits]).reshape(t.shape[0], -1)
    return t[torch.from_numpy(inst).to(dev)]


def _exact_picks(p, u):
    """The first completion whose running sum passes u times the whole, sums in order."""
    c = np.cumsum(p, axis=1)
    hit = c > (u * c[:, -1])[:, None]
    return torch.from_numpy(np.where(hit.any(1), hit.argmax(1), p.shape[1] - 1).astype(np.int64))


def _exact_fidelity(case, seed):
    a = _run_amplitudes(case, seed).to(_device())
    k, n = case["rows"], case["qubits"]
    x = (a[:, 0] * a[:, 0] + a[:, 1] * a[:, 1]) * 2.0 ** n
    mean, var = float(x.mean()), float(x.var(unbiased=False))
    f = min(max(mean - 1, 0.0), 1 - 1e-12)
    for _ in range(100):
        g = (x - 1) / (1 + f * (x - 1))
        f, old = min(max(f + float(g.sum() / (g * g).sum()), 0.0), 1 - 1e-12), f
        if abs(f - old) < 1e-14:
            break
    g = (x - 1) / (1 + f * (x - 1))
    q = torch.floor(x / (8.0 / case["bins"])).clamp(max=case["bins"]).to(torch.int64)
    return {"xeb": torch.tensor([mean - 1], dtype=torch.float64), "counts": torch.bincount(q, minlength=case["bins"] + 1),
            "fit": {"fidelity": f, "stderr": float((g * g).sum() ** -0.5),
                    "loglik": float(torch.log(1 + f * (x - 1)).sum() - x.sum()), "linear": mean - 1,
                    "linear_stderr": math.sqrt(var / k)}}


def _exact_mlp(case, seed):
    p, X, t, m, v = (x.to(_device()) for x in _mlp_inputs(case, seed))
    train = case["kind"] == "mlp_train"
    p, X, t, m, v = (p if train else p.half()).double(), X.double(), t.double(), m.double(), v.double()
    p.requires_grad_(train)
    w1, b1, w2, b2, w3, b3 = torch.split(p, [H * D, H, H * H, H, H, 1])
    y = torch.relu(torch.relu(X @ w1.view(H, D).T + b1) @ w2.view(H, H).T + b2) @ w3 + b3
    if not train:
        return y
    loss = ((y - t) ** 2).mean()
    g, = torch.autograd.grad(loss, p)
    # the entry point takes its constants in 32 bits
    lr, c1, c2, eps = (float(np.float32(c)) for c in (2e-3, 0.9, 0.999, 1e-8))
    m, v = c1 * m + (1 - c1) * g, c2 * v + (1 - c2) * g * g
    step = lr * (m / (1 - c1 ** 201)) / (torch.sqrt(v / (1 - c2 ** 201)) + eps)
    return {"params": (p - step).detach(), "m": m, "v": v, "grad": g, "loss": loss.detach().reshape(1)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sample":
        a = _batch_amplitudes(case, seed).numpy().reshape(case["rows"], -1, 2)
        return _exact_picks(a[..., 0] * a[..., 0] + a[..., 1] * a[..., 1], np.random.default_rng(int(seed)).random(case["rows"]))
    if kind == "fidelity":
        return _exact_fidelity(case, seed)
    if kind.startswith("mlp"):
        return _exact_mlp(case, seed)
    circ, _, struct, ssa, sliced = _network(_key(case))
    n, r = circ.n_qubits, case.get("open", 0)
    bits = _bits(case, n, seed)
    if kind == "slices":
        got = []
        for i in _slice_ids(case, seed, len(sliced))[:EXACT_SLICES]:
            fixed = {int(e): (int(i) >> j) & 1 for j, e in enumerate(sliced)}
            got.append(_contract(circ, ssa, bits, fixed)[:, 0])
        return [_real(torch.stack(got)), None]
    if not _whole(case):
        if sliced:
            return None
        got = _contract(circ, ssa, bits[:EXACT_ROWS], {}, _open_qubits(n, r))
        return [_real(got), None] + ([None] if r else [])
    psi = _state(circ)
    if kind == "stream":
        return [psi[_index(_bits(case, n, seed, b)).to(psi.device)].cpu().numpy().reshape(-1) for b in range(case["batches"])]
    base = _index(bits) & ~((1 << r) - 1)  # the open qubits are the lowest bits
    got = psi[(base[:, None] + torch.arange(1 << r)).to(psi.device)]
    return [_real(got)] + ([None] if r else [])
