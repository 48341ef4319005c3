"""The schedule that the tensor-core GEMM takes by rule (a group's whole B
resident, or one column tile's): the plan's own choice against both forced
schedules, on steps around the rule's edges.

Held to the 1e-4 of the BF16x3 form against the state vector.
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


def _tc(st):
    return st["mb"] >= 6 and st["kb"] >= 3 and not (st["mb"] + st["nb"] <= 5)


def _chunks(st):
    """B chunks resident under the two schedules: a group's, a column tile's."""
    nch = max(1, (1 << st["kb"]) // 16)
    return nch * (((st["max_group"] << st["nb"]) + 63) // 64), nch


# (layout, cycles, rows, tree seed, tree, whether a step is on the rule's side);
# instances of 1 to 16 columns in the others: the runs of the max fold
@pytest.mark.parametrize("layout,cycles,rows,seed,tree,rule", [
    ((4, 5), 10, 200, 2, 0, True), ((4, 5), 10, 200, 2, 4, True), ((4, 5), 10, 1000, 3, 1, True),
    ((3, 6), 12, 3000, 3, 3, True), ((4, 4), 12, 500, 2, 0, False), ((4, 4), 12, 500, 2, 2, False),
    ((4, 4), 12, 500, 2, 3, False), ((4, 4), 12, 3000, 2, 2, False)])
@pytest.mark.parametrize("rescale", [0, 1])
def test_rule_against_both_schedules(layout, cycles, rows, seed, tree, rule, rescale):
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    ref = sv.amplitudes(c, bits)
    got, p = run_plan(c, bits, ssa, precision="bf16x3", rescale=rescale)
    sides = [6 < _chunks(st)[0] <= 11 and _chunks(st)[1] <= 6 for st in p.tn_plan_steps() if _tc(st)]
    assert any(sides) == rule
    assert rel_l2(got, ref) <= 1e-4
    for cfg in (2, 3):  # every other step as the plan has it
        forced, _ = run_plan(c, bits, ssa, precision="bf16x3", rescale=rescale,
                             force_config=lambda st: cfg if _tc(st) and st["kernel"] == 1 else None)
        assert rel_l2(forced, ref) <= 1e-4


@pytest.mark.parametrize("layout,cycles,rows,seed,tree,many", [((4, 4), 12, 500, 3, 2, True), ((3, 6), 12, 37, 3, 0, False)])
@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
def test_tiles_of_16_columns(layout, cycles, rows, seed, tree, many, prec):
    # groups of 16 columns whose rows are neighbours in C: stored from registers
    # (few tiles a CTA) or staged (eight and more)
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=2)[tree]
    got, p = run_plan(c, bits, ssa, precision=prec)
    tiles = [st["n_groups"] << (st["mb"] - 7) for st, f in zip(p.tn_plan_steps(), p.tn_plan_step_forms())
             if f == tn.TN_FORM_TC and st["max_group"] << st["nb"] == 16 and st["mb"] >= 7
             and list(st["c_pos_m"][:2]) == [0, 1]]
    assert tiles and any(t >= 8 * 152 for t in tiles) == many
    assert rel_l2(got, sv.amplitudes(c, bits)) <= {"bf16x3": 1e-4, "tf32": 2e-2}[prec]
