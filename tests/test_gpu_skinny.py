"""Steps with few outputs per instance and a long K (the root with its open
qubits, and the steps just below it): every split of rows and columns that
the skinny kernel takes, against the state vector.

FP32 sums: held to the 1e-5 of the FP32 form.
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


def _takes(st):
    return st["kb"] >= 6 and st["nb"] <= 3 and st["mb"] + st["nb"] <= 5


@pytest.mark.parametrize("rescale", [0, 1])
@pytest.mark.parametrize("layout,open_q,tree", [
    ((4, 4), [], 1), ((4, 4), [15], 1), ((4, 4), [0, 15], 1), ((4, 4), [14, 15], 1), ((4, 4), [0, 1, 15], 1),
    ((4, 4), [12, 13, 14, 15], 1), ((4, 4), [11, 13, 14, 15], 1), ((4, 4), [0, 5, 8, 14, 15], 1),
    ((4, 4), [0, 1, 2, 3, 4], 1), ((4, 4), [12, 13, 14, 15], 2), ((4, 4), [0, 1, 2, 3, 4], 2),
    ((4, 5), [], 2), ((4, 5), [19], 2), ((4, 5), [0, 19], 2), ((4, 5), [0, 1], 2), ((4, 5), [16, 17, 18, 19], 2)])
def test_few_outputs_long_k(layout, open_q, tree, rescale):
    c = random_circuit(grid_layout(*layout), 12, seed=21)
    n = c.n_qubits
    bits = uniform_bitstrings(n, 37, seed=5)
    ssa = candidate_trees(network_structure(c), 37, seed=2, trials=2)[tree]
    got, p = run_plan(c, bits, ssa, precision="fp32", open_qubits=open_q, rescale=rescale,
                      force_kernel=lambda st: 1 if _takes(st) else None)
    takes = np.array([_takes(st) for st in p.tn_plan_steps()])
    assert np.any(takes) and np.all(p.tn_plan_step_forms()[takes] == tn.TN_FORM_SKINNY)
    r = len(open_q)
    ref = np.zeros((len(bits), 1 << r), np.complex128)
    for x in range(1 << r):
        b = bits.copy()
        for i, q in enumerate(sorted(open_q)):
            b[:, q] = (x >> (r - 1 - i)) & 1
        ref[:, x] = sv.amplitudes(c, b)
    assert rel_l2(got.reshape(ref.shape), ref) <= 1e-5
