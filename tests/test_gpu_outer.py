"""Grouped steps that leave the GEMM tiles where that fills the chip: short rows and many columns (K up to
32, N >= 32), and rows of 32 and more with few columns per A instance, from
the smallest M that each takes, against the state vector.

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


def _outer(st):
    return st["kb"] <= 5 and st["nb"] >= 5 and st["mb"] >= 5


def _narrow(st):
    return (st["kb"] >= 5 and st["mb"] >= 7 and (st["n_inst"] << st["nb"]) <= 16 * st["n_groups"] and
            (st["n_groups"] << (st["mb"] - 7)) >= 304)


# (layout, cycles, rows, tree seed, tree, step, kind)
@pytest.mark.parametrize("layout,cycles,rows,seed,tree,step,kind", [
    ((4, 4), 12, 37, 2, 4, 57, _outer), ((4, 4), 12, 3000, 3, 3, 57, _outer), ((4, 4), 10, 37, 4, 2, 50, _outer),
    ((4, 5), 10, 37, 2, 5, 70, _outer), ((4, 4), 12, 3000, 4, 4, 58, _outer), ((4, 5), 12, 37, 2, 4, 75, _outer),
    ((4, 4), 12, 500, 2, 0, 58, _outer), ((4, 4), 10, 500, 3, 3, 46, _outer), ((4, 5), 10, 3000, 2, 3, 70, _outer),
    ((4, 4), 12, 37, 2, 2, 58, _outer), ((4, 4), 12, 37, 4, 3, 62, _outer), ((4, 4), 12, 500, 3, 3, 60, _outer),
    ((4, 4), 12, 500, 4, 2, 53, _outer), ((4, 4), 12, 3000, 3, 3, 61, _outer), ((4, 4), 12, 37, 2, 2, 63, _outer),
    ((3, 6), 12, 37, 3, 2, 63, _outer), ((2, 8), 12, 37, 3, 0, 58, _outer), ((2, 8), 12, 500, 3, 1, 59, _outer),
    ((2, 8), 12, 3000, 3, 3, 57, _outer), ((4, 4), 12, 37, 2, 1, 63, _outer), ((2, 8), 10, 37, 3, 2, 48, _outer),
    ((2, 8), 10, 3000, 4, 2, 52, _outer), ((4, 5), 10, 37, 2, 5, 71, _outer), ((4, 4), 12, 37, 2, 4, 60, _outer),
    ((5, 4), 10, 37, 2, 4, 66, _outer), ((5, 4), 12, 500, 3, 3, 82, _outer), ((3, 6), 12, 500, 2, 0, 73, _outer),
    ((4, 4), 12, 37, 2, 4, 67, _narrow),
    ((4, 4), 12, 500, 3, 3, 69, _narrow), ((4, 4), 12, 3000, 3, 3, 66, _narrow), ((4, 5), 10, 37, 2, 2, 72, _narrow),
    ((4, 5), 12, 500, 2, 5, 89, _narrow), ((4, 5), 12, 3000, 3, 1, 87, _narrow)])
@pytest.mark.parametrize("prec,rescale", [("fp32", 0), ("fp32", 1), ("bf16x3", 1)])
def test_steps_off_the_gemm_tiles(layout, cycles, rows, seed, tree, step, kind, prec, rescale):
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    got, p = run_plan(c, bits, ssa, precision=prec, rescale=rescale,
                      force_config=lambda st: 2 if _outer(st) or _narrow(st) else None)
    st = p.tn_plan_steps()[step]
    form = p.tn_plan_step_forms()[step]
    want = tn.TN_FORM_NARROW
    if kind is _outer:  # not for few blocks, from K = 8 on
        ctab = st["n_groups"] if st["max_group"] << st["nb"] <= 64 else (st["n_inst"] << st["nb"]) // 64
        rows = min(1 << st["mb"], 256) * (2 if st["mb"] >= 9 and st["kb"] <= 4 else 1)
        blocks = ctab * ((1 << st["mb"]) // rows)
        takes = st["kb"] <= 2 or blocks >= (32 if st["kb"] == 5 else 48)
        want = tn.TN_FORM_OUTER if takes else tn.TN_FORM_SIMT
    if prec == "bf16x3" and st["kb"] >= 3 and st["mb"] >= 6:  # tensor cores, unless B is streamed for few columns
        streams_few = st["kb"] >= 8 and (st["n_inst"] << st["nb"]) <= 8 * st["n_groups"]
        want = tn.TN_FORM_NARROW if kind is _narrow and streams_few else tn.TN_FORM_TC
    assert form == want
    assert rel_l2(got, sv.amplitudes(c, bits)) <= {"fp32": 1e-5, "bf16x3": 1e-4}[prec]
