"""FP32 steps on the tensor cores (FP16x3: operands as scaled fp16 halves,
three products, units of 32 or 64 real k summed in FP32): plans with steps that
it takes, M = 64 to 2^16, K = 64 to 1024, N = 16 to 2^11, shared and separate
A instances, against the state vector.

Bounds: the 1e-5 of the FP32 form, and no more than the same plan has with
those steps on the FMA kernel (configuration 3).  Per product the split
leaves 2^-23 of each operand and drops 2^-22 of the product, both random; a
unit of 4 accumulations truncates 4 x 2^-24; the FMA kernel rounds 2 K times.
The bound on the ratio leaves 10 % for the two forms' different sums.
"""

import pytest

from gpu_helpers import rel_l2, run_plan
from oracle import sv
from rqc import grid_layout, network_structure, random_circuit
from rqc.bitstrings import uniform_bitstrings
from rqc.tree import candidate_trees

pytestmark = pytest.mark.gpu


def _takes(st):
    return st["mb"] >= 6 and st["kb"] >= 6 and (st["nb"] >= 6 or (st["n_inst"] << st["nb"]) >= 32 * st["n_groups"])


@pytest.mark.parametrize("layout,cycles,rows,seed,tree", [
    ((4, 4), 12, 37, 2, 1), ((4, 4), 12, 37, 4, 3), ((4, 4), 12, 500, 4, 4), ((4, 4), 12, 3000, 3, 3),
    ((4, 5), 10, 37, 3, 3), ((4, 5), 12, 37, 2, 3), ((4, 5), 12, 37, 4, 1), ((4, 5), 12, 500, 2, 4),
    ((4, 5), 12, 500, 3, 3), ((4, 5), 12, 37, 4, 3), ((3, 6), 12, 37, 3, 2), ((4, 4), 14, 500, 2, 3), ((4, 4), 14, 3000, 4, 3)])
def test_error_is_that_of_fp32(layout, cycles, rows, seed, tree):
    c = random_circuit(grid_layout(*layout), cycles, seed=21)
    bits = uniform_bitstrings(c.n_qubits, rows, seed=5)
    ssa = candidate_trees(network_structure(c), rows, seed=seed, trials=3)[tree]
    ref = sv.amplitudes(c, bits)
    got, p = run_plan(c, bits, ssa, precision="fp32")
    assert any(_takes(st) for st in p.tn_plan_steps())
    fma, _ = run_plan(c, bits, ssa, precision="fp32", force_config=lambda st: 3 if _takes(st) else None)
    err, own = rel_l2(got, ref), rel_l2(fma, ref)
    assert own <= 1e-5 and err <= 1.1 * own
    plain, _ = run_plan(c, bits, ssa, precision="fp32", rescale=0)  # no maxima, no scales: the FMA kernel
    assert rel_l2(plain, ref) <= 1e-5
