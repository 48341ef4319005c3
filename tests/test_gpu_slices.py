"""Single slices of a batched plan: a pass computes only the instances of the
slice asked for, and keeps what no changed slice value touches.  Every slice,
asked for alone, out of order, several of a batch and all of it, against the
partials of a plan that runs one slice per pass.

The same kernels on the same operands: FP32 sums in another split at most,
held to 2e-6; BF16x3 to 1e-4 of each other.
"""

import numpy as np
import pytest

from gpu_helpers import rel_l2, require_cuda
from rqc import grid_layout, network_structure, random_circuit
from rqc.bitstrings import uniform_bitstrings
from rqc.tree import ContractionTree, candidate_trees, choose_slices

pytestmark = pytest.mark.gpu


def _partials(tn, torch, c, bits, ssa, sl, ids, prec, low, force=None, calls=1, **opts):
    p = tn.Plan(c, bits, ssa, sl, slice_batch_log2=low, **opts)
    if force is not None:
        for s, st in enumerate(p.tn_plan_steps()):
            if force(st) is not None:
                p.tn_plan_set_config(s, force(st))
    ws = torch.full((max(p.info["workspace_bytes"], 256),), 255, dtype=torch.uint8, device="cuda")  # NaN everywhere
    stream = torch.cuda.current_stream()
    p.tn_plan_bind(ws, stream=stream)
    n = len(bits) * p.info["amps_per_row"]
    out = torch.zeros(len(ids), 2 * n, dtype=torch.float64, device="cuda")
    per = -(-len(ids) // calls)
    for k in range(0, len(ids), per):
        p.tn_contract_slices(ids[k:k + per], out[k:k + per], prec, stream=stream)
    p.tn_plan_check(stream=stream)
    return out.cpu().numpy().view(np.complex128), p


@pytest.mark.parametrize("prec,config", [("fp32", None), ("fp32", 1), ("fp32", 3), ("bf16x3", 2), ("bf16x3", 3)])
@pytest.mark.parametrize("layout,cycles,rows,tree,n_sliced,low,opts", [
    ((4, 4), 10, 300, 1, 5, 3, {}), ((4, 5), 10, 90, 2, 4, 2, {"rescale": 0}),
    ((4, 5), 14, 60, 1, 4, 3, {}),  # steps long enough that two slices of eight still run one by one
    ((4, 4), 10, 40, 3, 4, 4, {"open_qubits": [0, 15]}), ((4, 4), 10, 200, 0, 5, 2, {"fuse": 1, "fuse_max_bits": 8})])
def test_slices_alone_match_whole_passes(layout, cycles, rows, tree, n_sliced, low, opts, prec, config):
    torch, tn = require_cuda()
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    st = network_structure(c)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(st, rows, seed=2, trials=2)[tree]
    sl = choose_slices(st, ContractionTree(ssa=ssa), rows, n_sliced=n_sliced)
    row_ok = lambda s: s["nb"] <= 4 and s["kb"] + s["nb"] <= 8  # noqa: E731
    force = None if config is None else (lambda s: config if config >= 2 or row_ok(s) else None)
    n = 1 << n_sliced
    ids = np.random.default_rng(3).permutation(n)
    ref, _ = _partials(tn, torch, c, bits, ssa, sl, ids, prec, 0, force, **opts)
    tol = 2e-6 if prec == "fp32" else 1e-4
    # one slice a call; a few at a time (some batches in part, some by more
    # than half); all at once (whole passes)
    for calls in (n, 4, 1):
        got, p = _partials(tn, torch, c, bits, ssa, sl, ids, prec, low, force, calls, **opts)
        assert p.info["slice_batch_log2"] == low
        assert rel_l2(got, ref) <= tol, calls
    few = ids[:3]  # a call whose slices lie far apart
    got, _ = _partials(tn, torch, c, bits, ssa, sl, few, prec, low, force, **opts)
    assert rel_l2(got, ref[:3]) <= tol


@pytest.mark.parametrize("layout,cycles,rows,tree", [((3, 4), 8, 64, 1), ((4, 4), 10, 300, 1), ((4, 5), 10, 90, 2)])
def test_some_slices_of_a_small_plan_take_no_longer_than_all(layout, cycles, rows, tree):
    # launches and merged steps set the time of these plans: a pass per slice
    # would take as often as long as a whole pass
    torch, tn = require_cuda()
    import time
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    st = network_structure(c)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(st, rows, seed=2, trials=3)[tree]
    sl = choose_slices(st, ContractionTree(ssa=ssa), rows, n_sliced=3)
    p = tn.Plan(c, bits, ssa, sl, slice_batch_log2=3)
    ws = torch.empty(p.info["workspace_bytes"], dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream()
    p.tn_plan_bind(ws, stream=stream)
    out = torch.zeros(8, 2 * rows, dtype=torch.float64, device="cuda")

    def seconds(n):
        t = []
        for _ in range(20):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            p.tn_contract_slices(np.arange(n), out[:n], "fp32", stream=stream)
            torch.cuda.synchronize()
            t.append(time.perf_counter() - t0)
        return float(np.median(t))

    whole = seconds(8)
    assert seconds(4) <= 1.3 * whole and seconds(2) <= 1.3 * whole and seconds(1) <= 1.3 * whole
    assert layout == (3, 4) or tn.TN_FORM_FEW in p.tn_plan_step_forms()  # on one slice's instances
