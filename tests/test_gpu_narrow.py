"""Steps with rows of 32 to 128 entries and few columns per A instance: the
row kernel's tiles of 8 and of 16 columns, groups of fewer columns than a
tile, of a few tiles and of more than 64, against the state vector.

FP32 sums: held to the 1e-5 of the FP32 form.
"""

import pytest

from gpu_helpers import rel_l2, run_plan
from oracle import sv
from paper_2212_04749_gb300 import tn
from rqc import grid_layout, network_structure, random_circuit
from rqc.bitstrings import uniform_bitstrings
from rqc.tree import candidate_trees

pytestmark = pytest.mark.gpu


def _takes(st):
    return st["mb"] >= 7 and st["kb"] >= 5 and st["kb"] + st["nb"] <= 8 and st["nb"] <= 4


# (layout, cycles, rows, tree seed, tree, step, columns per A instance above 8, groups above 16 columns)
@pytest.mark.parametrize("layout,cycles,rows,seed,tree,step,wide,many", [
    ((4, 4), 12, 37, 2, 2, 67, False, False), ((4, 4), 12, 500, 3, 2, 66, True, True),
    ((4, 4), 12, 500, 3, 2, 67, True, False), ((4, 4), 12, 3000, 3, 3, 67, False, False),
    ((4, 4), 12, 3000, 3, 3, 68, True, True), ((4, 4), 10, 37, 4, 2, 53, True, True),
    ((4, 4), 10, 500, 2, 1, 55, True, True), ((4, 4), 10, 500, 3, 3, 56, True, True),
    ((4, 5), 10, 37, 4, 0, 73, False, True), ((4, 5), 10, 500, 2, 4, 74, False, False),
    ((4, 5), 12, 3000, 4, 3, 88, True, False), ((4, 5), 12, 3000, 3, 2, 89, False, False)])
@pytest.mark.parametrize("rescale", [0, 1])
def test_tiles_of_columns(layout, cycles, rows, seed, tree, step, wide, many, rescale):
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    got, p = run_plan(c, bits, ssa, precision="fp32", rescale=rescale,
                      force_kernel=lambda st: 0 if _takes(st) else None)
    st = p.tn_plan_steps()[step]
    assert p.tn_plan_step_forms()[step] == tn.TN_FORM_NARROW
    assert ((st["n_inst"] << st["nb"]) > 8 * st["n_groups"], (st["max_group"] << st["nb"]) > 16) == (wide, many)
    assert rel_l2(got, sv.amplitudes(c, bits)) <= 1e-5
