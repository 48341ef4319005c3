"""Fused chains over tile sizes and step shapes: every chain set to run as its
kernel, against the state vector, with tiles of 2^5 to 2^12 entries, steps of
K up to 64 and N up to 16 whose rows are more and fewer than the block's
threads, several instances, slices, open qubits, with and without the
rescale; and the chains that a plan without the fuse option makes of its
streaming steps, against the same steps one by one.

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
    c = random_circuit(grid_layout(*layout), cycles, seed=41)
    st = network_structure(c)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=6)
    ssa = candidate_trees(st, rows, seed=4, trials=3)[tree]
    sl = choose_slices(st, ContractionTree(ssa=ssa), rows, n_sliced=n_sliced) if n_sliced else []
    return c, bits, ssa, sl


def _run(tn, torch, p, n):
    ws = torch.empty(max(p.info["workspace_bytes"], 256), dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream()
    p.tn_plan_bind(ws, stream=st)
    amps = torch.zeros(2 * n, dtype=torch.float64, device="cuda")
    p.tn_contract(amps, "fp32", stream=st)
    p.tn_plan_check(stream=st)
    return amps.cpu().numpy().view(np.complex128), p.tn_plan_step_times()[1]


@pytest.mark.parametrize("rescale", [0, 1])
@pytest.mark.parametrize("bits_max", [3, 6, 8, 10])
@pytest.mark.parametrize("layout,cycles,rows,tree,n_sliced,open_q", [
    ((3, 4), 8, 64, 1, 0, []), ((4, 4), 9, 300, 0, 0, []), ((4, 4), 9, 300, 2, 3, []), ((4, 4), 11, 50, 4, 0, [0, 9, 15]),
    ((4, 5), 9, 200, 1, 0, [])])
def test_chains_set_to_their_kernel(layout, cycles, rows, tree, n_sliced, open_q, bits_max, rescale):
    torch, tn = require_cuda()
    c, bits, ssa, sl = _case(layout, cycles, rows, tree, n_sliced)
    p = tn.Plan(c, bits, ssa, sl, fuse=1, fuse_max_bits=bits_max, rescale=rescale, open_qubits=open_q)
    if p.info["n_chains"] == 0:
        pytest.skip("no chain touches so few bits")
    for ch in range(p.info["n_chains"]):
        p.tn_plan_set_chain(ch, 1)
    r = len(open_q)
    got, kinds = _run(tn, torch, p, rows << r)
    steps = p.tn_plan_steps()
    assert all(k == 3 for s, k in zip(steps, kinds) if s["chain"] >= 0)
    ref = np.zeros((rows, 1 << r), np.complex128)
    for x in range(1 << r):
        b = bits.copy()
        for i, q in enumerate(open_q):
            b[:, q] = (x >> (r - 1 - i)) & 1
        ref[:, x] = sv.amplitudes(c, b)
    assert rel_l2(got.reshape(ref.shape), ref) <= 1e-5


@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
@pytest.mark.parametrize("layout,cycles,rows,tree,n_sliced", [((4, 5), 12, 700, 0, 0), ((4, 5), 12, 700, 1, 2),
                                                              ((4, 5), 8, 33, 2, 0), ((3, 6), 10, 5, 0, 1)])
def test_streaming_steps_without_the_fuse_option(layout, cycles, rows, tree, n_sliced, prec):
    c, bits, ssa, sl = _case(layout, cycles, rows, tree, n_sliced)
    ref = sv.amplitudes(c, bits)
    tol = {"fp32": 1e-5, "bf16x3": 1e-3}[prec]
    got, p = run_plan(c, bits, ssa, sl, precision=prec)
    assert p.info["n_chains"] == 0 and all(s["chain"] == -1 for s in p.tn_plan_steps())
    assert rel_l2(got, ref) <= tol
    base = p.tn_plan_get_configs()
    row = lambda st: 0 if st["nb"] <= 4 and st["kb"] + st["nb"] <= 8 else 2  # noqa: E731
    got1, p1 = run_plan(c, bits, ssa, sl, precision=prec, force_config=row)
    assert not np.any(p1.tn_plan_step_times()[1] == 3)  # kernels chosen step by step: none fused
    assert rel_l2(got1, ref) <= tol
    if (layout, tree) == ((4, 5), 0):
        assert np.sum(p.tn_plan_step_times()[1] == 3) >= 4
    assert np.array_equal(base, p.tn_plan_get_configs())


@pytest.mark.parametrize("log2,layers", [(30, 2), (60, 1)])
@pytest.mark.parametrize("fuse,config", [(0, None), (1, None), (0, 0), (0, 2)])
@pytest.mark.parametrize("layout,cycles,rows,tree,n_sliced", [((4, 5), 12, 700, 0, 0), ((4, 5), 12, 700, 1, 2)])
def test_operands_of_any_scale(layout, cycles, rows, tree, n_sliced, fuse, config, log2, layers):
    # gates of 2^-log2 in some layers and of 2^log2 in the next: a few of them
    # leave the range of FP32.  The rescale keeps every intermediate in range,
    # step by step and within a fused chain
    c, bits, ssa, sl = _case(layout, cycles, rows, tree, n_sliced)
    for g in c.two_qubit_gates:
        g.matrix = g.matrix * 2.0 ** (log2 if (g.layer // 2 // layers) % 2 else -log2)
    ref = sv.amplitudes(c, bits)
    row = lambda st: config if config != 0 or st["nb"] <= 4 and st["kb"] + st["nb"] <= 8 else 2  # noqa: E731
    got, p = run_plan(c, bits, ssa, sl, fuse=fuse, force_config=None if config is None else row)
    assert np.any(p.tn_plan_step_forms() == 3) == (config is None)
    assert rel_l2(got, ref) <= 1e-5
