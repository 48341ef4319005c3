"""FP32 steps on the tensor cores (BF16x6: operands as three bf16 parts, six
products, units of 32 or 64 real k summed in FP32): plans with steps that
it takes, M = 64 to 2^16, K = 64 to 1024, N = 16 to 2^11, shared and separate
A instances, against the state vector.

Bounds: the 1e-5 of the FP32 form, and no more than the same plan has with
those steps on the FMA kernel (configuration 3).  The parts hold every bit of
an operand; the three products left out are below 2^-24 of the whole; a
unit's large products are added in 2 to 4 accumulations that truncate; the FMA
kernel rounds 2 K times.  Most of a plan's error comes from its other steps,
which both arms share; the bound on the ratio leaves 10 % for the two forms'
different rounding.
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


def _both(c, bits, ssa):
    """Amplitudes with the plan's own FP32 kernels and with the steps that
    went to the tensor cores on FMAs (configuration 3)."""
    got, p = run_plan(c, bits, ssa, precision="fp32")
    on_tc = p.tn_plan_step_forms() == tn.TN_FORM_TC_FP32
    assert np.any(on_tc)
    own = iter(on_tc)
    fma, q = run_plan(c, bits, ssa, precision="fp32", force_config=lambda st: 3 if next(own) else None)
    assert not np.any(np.isin(q.tn_plan_step_forms(), (tn.TN_FORM_TC_FP32, tn.TN_FORM_TC)))
    return got, fma


@pytest.mark.parametrize("layout,cycles,rows,seed,tree", [
    ((4, 4), 12, 37, 2, 1), ((4, 4), 12, 37, 4, 3), ((4, 4), 12, 500, 4, 4), ((4, 4), 12, 3000, 3, 3),
    ((4, 5), 10, 37, 3, 3), ((4, 5), 12, 37, 2, 3), ((4, 5), 12, 37, 4, 1), ((4, 5), 12, 500, 2, 4),
    ((4, 5), 12, 500, 3, 3), ((4, 5), 12, 37, 4, 3), ((3, 6), 12, 37, 3, 2), ((4, 4), 14, 500, 2, 3), ((4, 4), 14, 3000, 4, 3)])
def test_error_is_that_of_fp32(layout, cycles, rows, seed, tree):
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    ref = sv.amplitudes(c, bits)
    got, fma = _both(c, bits, ssa)
    err, own = rel_l2(got, ref), rel_l2(fma, ref)
    assert own <= 1e-5 and err <= 1.1 * own
    plain, p = run_plan(c, bits, ssa, precision="fp32", rescale=0)  # no maxima, no scales: the FMA kernel
    assert not np.any(p.tn_plan_step_forms() == tn.TN_FORM_TC_FP32)
    assert rel_l2(plain, ref) <= 1e-5


def _wide_range(layout, cycles, at, qubits, log2):
    """A random circuit whose state after two-qubit layer `at` has |1> of
    each of `qubits` scaled by 2^-log2; the next two-qubit gate on the qubit
    projects on |1> and scales back.  Tensors between the two hold entries
    2^-log2 apart for every such bond, and only the small ones reach the
    amplitudes."""
    c = random_circuit(layout, cycles, seed=21)

    def on(gate, q, d0, d1):
        return np.diag([(d0, d1)[(x >> (1 if gate.qubits[0] == q else 0)) & 1] for x in range(4)])

    for q in qubits:
        mine = [g for g in c.gates if q in g.qubits]
        two = [i for i, g in enumerate(mine) if len(g.qubits) == 2]
        i = max(j for j in two if mine[j].layer <= 2 * at + 1)
        n = min(j for j in two if j > i)
        for g in mine[i + 1:n]:
            g.matrix = np.eye(2, dtype=complex)
        mine[i].matrix = on(mine[i], q, 1.0, 2.0 ** -log2) @ mine[i].matrix
        mine[n].matrix = mine[n].matrix @ on(mine[n], q, 0.0, 2.0 ** log2)
    return c


@pytest.mark.parametrize("layout,cycles,rows,seed,tree", [
    ((4, 4), 12, 500, 4, 4), ((4, 4), 12, 3000, 3, 3), ((4, 5), 10, 37, 3, 3), ((4, 5), 12, 37, 2, 3),
    ((4, 5), 12, 500, 3, 3), ((3, 6), 12, 37, 3, 2)])
@pytest.mark.parametrize("at", [4, 6])
def test_small_entries_beside_large_ones_keep_their_bits(layout, cycles, rows, seed, tree, at):
    # 2^-10 for each of 8 qubits: the entries that count are down to 2^-80 of
    # their instance's largest
    lay = grid_layout(*layout)
    c = _wide_range(lay, cycles, at, range(0, 2 * 8, 2), 10)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    ref = sv.amplitudes(c, bits)
    got, fma = _both(c, bits, ssa)
    err, own = rel_l2(got, ref), rel_l2(fma, ref)
    assert own <= 1e-5 and err <= 1.1 * own
