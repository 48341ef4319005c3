"""Steps of few multiply-adds run by themselves (too many for the merged
launches): an output per thread or per few lanes, over plans whose steps take
K = 1 to 2^10, one and many instances, instances smaller and larger than a
block, against the state vector.

FP32 sums: held to the 1e-5 of the FP32 form; BF16x3 to its 1e-4.
"""

import numpy as np
import pytest

from gpu_helpers import rel_l2, run_plan
from oracle import sv
from paper_2212_04749_gb300 import tn
from rqc import grid_layout, network_structure, random_circuit
from rqc.bitstrings import uniform_bitstrings
from rqc.tree import candidate_trees

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,rescale,tol", [("fp32", 0, 1e-5), ("fp32", 1, 1e-5), ("bf16x3", 1, 1e-4)])
@pytest.mark.parametrize("layout,cycles,rows,seed,tree", [
    ((4, 4), 12, 37, 2, 1), ((4, 4), 12, 500, 2, 0), ((4, 4), 12, 3000, 3, 3), ((4, 4), 10, 37, 4, 2),
    ((4, 4), 10, 500, 3, 3), ((4, 5), 10, 37, 2, 5), ((4, 5), 10, 3000, 2, 3), ((3, 6), 12, 37, 3, 2),
    ((2, 8), 12, 37, 2, 0), ((2, 8), 12, 3000, 3, 3), ((3, 5), 10, 500, 2, 1), ((4, 4), 14, 3000, 4, 3)])
def test_steps_of_few_multiply_adds(layout, cycles, rows, seed, tree, prec, rescale, tol):
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    got, p = run_plan(c, bits, ssa, precision=prec, rescale=rescale)
    assert tn.TN_FORM_FEW in p.tn_plan_step_forms()
    assert rel_l2(got, sv.amplitudes(c, bits)) <= tol


@pytest.mark.parametrize("layout,cycles,rows,tree", [((4, 5), 12, 500, 0), ((3, 6), 12, 3000, 1), ((4, 5), 14, 37, 2)])
def test_larger_steps_leave_it_for_a_tuned_configuration(layout, cycles, rows, tree):
    # above 2^18 outputs: an output per thread in the place of the plan's own row
    # kernel, but the row kernel where its second schedule was chosen
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=3, trials=2)[tree]
    ref = sv.amplitudes(c, bits)
    got, p = run_plan(c, bits, ssa, precision="fp32")
    out = np.array([st["n_inst"] << (st["mb"] + st["nb"]) for st in p.tn_plan_steps()])
    big = (out > 1 << 18) & (p.tn_plan_step_forms() == tn.TN_FORM_FEW)
    big &= np.array([st["nb"] <= 4 and st["kb"] + st["nb"] <= 8 for st in p.tn_plan_steps()])
    assert np.any(big)
    own = iter(big)
    tuned, q = run_plan(c, bits, ssa, precision="fp32",
                        force_config=lambda st: 1 + tn.TN_CONFIG_TUNED if next(own) else None)
    assert np.all(np.isin(q.tn_plan_step_forms()[big], (tn.TN_FORM_ROW, tn.TN_FORM_NARROW)))
    assert rel_l2(got, ref) <= 1e-5 and rel_l2(tuned, ref) <= 1e-5
