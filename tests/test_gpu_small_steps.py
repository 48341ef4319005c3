"""Small steps that share launches: the merged launches against the state
vector, over circuits whose small steps have K = 1 to 64, single and many
instances per A, slices in one pass and in many, open qubits, with and
without the rescale, and in a workspace that gives their outputs no slots of
their own (the launch order then follows who overwrites whom).

FP32 sums: held to the 1e-5 of the FP32 form.
"""

import numpy as np
import pytest

from gpu_helpers import rel_l2, require_cuda, run_plan
from oracle import sv
from rqc import grid_layout, network_structure, random_circuit
from rqc.bitstrings import uniform_bitstrings
from rqc.tree import ContractionTree, candidate_trees, choose_slices

pytestmark = pytest.mark.gpu


def _case(layout, cycles, rows, tree, n_sliced):
    c = random_circuit(grid_layout(*layout), cycles, seed=31)
    st = network_structure(c)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=6)
    ssa = candidate_trees(st, rows, seed=4, trials=2)[tree]
    sl = choose_slices(st, ContractionTree(ssa=ssa), rows, n_sliced=n_sliced) if n_sliced else []
    return c, bits, ssa, sl


@pytest.mark.parametrize("rescale", [0, 1])
@pytest.mark.parametrize("layout,cycles,rows,tree,n_sliced,low", [
    ((3, 3), 5, 1, 0, 0, -1), ((3, 4), 8, 64, 1, 0, -1), ((3, 4), 8, 500, 2, 3, 1), ((4, 4), 9, 300, 3, 2, 0),
    ((4, 4), 7, 33, 0, 4, -1)])
def test_merged_small_steps_match_state_vector(layout, cycles, rows, tree, n_sliced, low, rescale):
    torch, tn = require_cuda()
    c, bits, ssa, sl = _case(layout, cycles, rows, tree, n_sliced)
    ref = sv.amplitudes(c, bits)
    got, p = run_plan(c, bits, ssa, sl, rescale=rescale, slice_batch_log2=low)
    kinds = p.tn_plan_step_times()[1]
    assert np.sum(kinds == 4) >= 4 and p.tn_plan_launches() < p.info["launches_per_call"]
    assert rel_l2(got, ref) <= 1e-5
    # one by one, each kernel set by hand: the same amplitudes
    got1, p1 = run_plan(c, bits, ssa, sl, rescale=rescale, slice_batch_log2=low,
                        force_config=lambda st: 1 if st["nb"] <= 4 and st["kb"] + st["nb"] <= 8 else 3)
    assert not np.any(p1.tn_plan_step_times()[1] == 4) and p1.tn_plan_launches() == p1.info["launches_per_call"]
    assert rel_l2(got, got1) <= 2e-6
    # a limit just below that workspace: no slots of their own
    kw = dict(rescale=rescale, slice_batch_log2=p.info["slice_batch_log2"])
    tight, q = run_plan(c, bits, ssa, sl, workspace_limit=p.info["workspace_bytes"] - 1, **kw)
    assert q.info["workspace_bytes"] < p.info["workspace_bytes"]
    assert np.any(q.tn_plan_step_times()[1] == 4)
    assert rel_l2(tight, ref) <= 1e-5


@pytest.mark.parametrize("open_q", [[0], [3, 11], [0, 5, 8, 14, 15]])
def test_merged_small_steps_with_open_qubits(open_q):
    c, bits, ssa, _ = _case((4, 4), 8, 20, 1, 0)
    got, p = run_plan(c, bits, ssa, open_qubits=open_q)
    assert np.any(p.tn_plan_step_times()[1] == 4)
    r = len(open_q)
    ref = np.zeros((len(bits), 1 << r), np.complex128)
    for x in range(1 << r):
        b = bits.copy()
        for i, q in enumerate(open_q):
            b[:, q] = (x >> (r - 1 - i)) & 1
        ref[:, x] = sv.amplitudes(c, b)
    assert rel_l2(got.reshape(ref.shape), ref) <= 1e-5


def test_small_chains_run_fused_where_chosen_and_merged_otherwise():
    # a chain of small steps shares the merged launches unless its fused
    # kernel is chosen; both give the same amplitudes
    torch, tn = require_cuda()
    c, bits, ssa, _ = _case((3, 4), 8, 64, 1, 0)
    ref = sv.amplitudes(c, bits)
    p = tn.Plan(c, bits, ssa, fuse=1, fuse_max_bits=7)
    n = p.info["n_chains"]
    assert n >= 2 and np.all(p.tn_plan_get_chains() == 1)
    ws = torch.empty(p.info["workspace_bytes"], dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream()
    p.tn_plan_bind(ws, stream=st)
    amps = torch.zeros(2 * len(bits), dtype=torch.float64, device="cuda")
    for on in (False, True):
        if on:
            for ch in range(n):
                p.tn_plan_set_chain(ch, 1)
        amps.zero_()
        p.tn_contract(amps, "fp32", stream=st)
        p.tn_plan_check(stream=st)
        assert np.any(p.tn_plan_step_times()[1] == 3) == on
        assert rel_l2(amps.cpu().numpy().view(np.complex128), ref) <= 1e-5
