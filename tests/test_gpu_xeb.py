"""Fidelity analysis on the GPU (linear XEB error bar, maximum-likelihood fit
to the Porter-Thomas mixture of Eq. (fxeb), histogram of x = N |amp|^2)
against the float64 oracle on the same amplitudes, and on amplitudes the
library contracted for bitstrings drawn from the exact distribution and
uniformly.

Tolerances: the device sums run in FP64 in another order than numpy's
(relative error ~1e-15 per sum), held to 1e-11; the fitted F follows the
sums, held to 1e-9; histogram bins are integer decisions taken by the same
correctly rounded FP64 operations on both sides, compared exactly.
"""

import numpy as np
import pytest

from gpu_helpers import require_cuda, run_plan
from oracle import sv
from oracle import xeb as oxeb

pytestmark = pytest.mark.gpu


def _amps(k, n, seed):
    # Porter-Thomas-like amplitudes: complex normal, |amp|^2 of mean 2^-n
    rng = np.random.default_rng(seed)
    return (rng.normal(size=k) + 1j * rng.normal(size=k)) * np.sqrt(0.5 / 2 ** n)


def _dev(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a, np.complex128).view(np.float64)).cuda()


@pytest.mark.parametrize("k", [1, 1000, 300001])
def test_moments_match_oracle(k):
    torch, tn = require_cuda()
    n = 24
    a = _amps(k, n, 1)
    d = _dev(torch, a)
    out = torch.empty(5, dtype=torch.float64, device="cuda")
    for f in (0.0, 0.37, 0.99):
        tn.tn_pt_moments(d, k, n, f, out)
        got = out.cpu().numpy()
        ref = oxeb.pt_moments(oxeb.x_values(a, n), f)
        assert np.all(np.abs(got - ref) <= 1e-11 * np.maximum(np.abs(ref), 1.0)), (f, got, ref)


def test_fit_matches_oracle_and_histogram_is_exact():
    torch, tn = require_cuda()
    from paper_2212_04749_gb300 import xeb
    n, k = 30, 200000
    rng = np.random.default_rng(4)
    # a mixture at F = 0.4: ideal samples have |amp|^2 size-biased (x e^-x)
    x = np.where(rng.random(k) < 0.4, rng.gamma(2.0, 1.0, k), rng.exponential(1.0, k))
    a = np.sqrt(x / 2 ** n) * np.exp(2j * np.pi * rng.random(k))
    d = _dev(torch, a)
    got = xeb.porter_thomas_fit(d, k, n)
    ref = oxeb.pt_fit(oxeb.x_values(a, n), start=got["linear"])
    assert abs(got["fidelity"] - ref["fidelity"]) < 1e-9
    assert abs(got["stderr"] - ref["stderr"]) < 1e-9 * ref["stderr"]
    assert abs(got["linear"] - ref["linear"]) < 1e-12
    assert abs(got["fidelity"] - 0.4) < 4 * got["stderr"]
    for x_max, nbins in ((8.0, 64), (5.0, 7), (1e-3, 1), (40.0, 8192)):
        h = xeb.porter_thomas_histogram(d, k, n, x_max=x_max, nbins=nbins)
        assert np.array_equal(h, oxeb.pt_histogram(oxeb.x_values(a, n), x_max, nbins)), (x_max, nbins)
    e = xeb.porter_thomas_expected(64, 8.0, k, got["fidelity"])
    h = xeb.porter_thomas_histogram(d, k, n)
    assert np.all(np.abs(h - e) < 5 * np.sqrt(e) + 5)


def test_fit_on_contracted_amplitudes():
    # 20 qubits, 20 cycles: bitstrings drawn from the exact output
    # distribution (oracle state vector) give F = 1, uniform ones F = 0,
    # each within 4 standard errors, from amplitudes the library contracted
    torch, tn = require_cuda()
    from paper_2212_04749_gb300 import xeb
    from rqc import grid_layout, network_structure, random_circuit
    from rqc.bitstrings import bitstrings_from_indices
    from rqc.tree import candidate_trees
    c = random_circuit(grid_layout(4, 5), 20, seed=77)
    psi = sv.state(c)
    p = np.abs(psi) ** 2
    rng = np.random.default_rng(9)
    k = 3000
    for f_true, idx in ((1.0, rng.choice(p.size, size=k, p=p / p.sum())), (0.0, rng.integers(0, p.size, size=k))):
        bits = bitstrings_from_indices(idx, 20)
        ssa = candidate_trees(network_structure(c), k, seed=2, trials=1)[0]
        amps, _ = run_plan(c, bits, ssa, [], precision="fp32")
        d = _dev(torch, amps)
        r = xeb.porter_thomas_fit(d, k, 20)
        print(f"F_true {f_true}: fit {r['fidelity']:.4f} +- {r['stderr']:.4f}, "
              f"linear {r['linear']:.4f} +- {r['linear_stderr']:.4f}")
        assert abs(r["fidelity"] - f_true) < 4 * r["stderr"] + 1e-6
        assert abs(r["linear"] - f_true) < 4 * r["linear_stderr"]


@pytest.mark.parametrize("k", [1, 511, 512, 2047, 2049, 8193, 20481, 1300003])
@pytest.mark.parametrize("f", [0.0, 0.37, 1.0 - 2.0 ** -53])
def test_moments_scratch_form_and_xeb_at_block_edges(k, f):
    # one block, part of a cluster, whole clusters, every SM; groups of four
    # amplitudes and their remainders; products of four 1 + F (x - 1) of
    # 1e-16 (x = 0 at F = 1 - 2^-53) and beyond the range of a double
    torch, tn = require_cuda()
    n = 20
    a = _amps(k, n, 3)
    a[: k // 7] = 0.0
    a[k // 7: k // 5] *= 1e60
    d = _dev(torch, a)
    x = oxeb.x_values(a, n)
    ref = oxeb.pt_moments(x, f)
    out = torch.full((5,), float("nan"), dtype=torch.float64, device="cuda")
    scratch = torch.empty(tn.tn_pt_moments_scratch_bytes(k), dtype=torch.uint8, device="cuda")
    for log in (True, False):
        tn.tn_pt_moments_scratch(d, k, n, f, out, scratch, want_log=log)
        got = out.cpu().numpy()
        want = ref if log else np.where(np.arange(5) == 2, 0.0, ref)
        assert np.all(np.abs(got - want) <= 1e-11 * np.maximum(np.abs(want), 1.0)), (f, log, got, want)
    tn.tn_pt_moments(d, k, n, f, out)
    assert np.all(np.abs(out.cpu().numpy() - ref) <= 1e-11 * np.maximum(np.abs(ref), 1.0))
    tn.tn_xeb(d, k, n, out)
    want = np.sum(np.abs(a) ** 2) * 2.0 ** n / k - 1.0
    assert abs(out[0].item() - want) <= 1e-12 * max(abs(want), 1.0)
    with pytest.raises(tn.TnError):
        tn.tn_pt_moments_scratch(d, k, n, f, out, scratch[:-1])


@pytest.mark.parametrize("kind", ["stream", "handle", "current"])
def test_analysis_on_a_stream_that_is_still_busy(kind):
    # the amplitudes arrive 50 ms late on a stream of their own: the sums and
    # counts read are those of the late amplitudes, from the first pass on
    torch, tn = require_cuda()
    from paper_2212_04749_gb300 import xeb
    n, k = 24, 50001
    d = _dev(torch, _amps(k, n, 6))
    fit, hist = xeb.porter_thomas_fit(d, k, n), xeb.porter_thomas_histogram(d, k, n)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    arg = {"stream": side, "handle": side.cuda_stream, "current": None}[kind]
    for f, want in ((xeb.porter_thomas_fit, fit), (xeb.porter_thomas_histogram, hist)):
        with torch.cuda.stream(side):
            late = torch.zeros_like(d)
            torch.cuda._sleep(100_000_000)
            late.copy_(d)
        with torch.cuda.stream(side if kind == "current" else torch.cuda.default_stream()):
            got = f(late, k, n, stream=arg)
        assert np.array_equal(got, want) if isinstance(want, np.ndarray) else got == want


@pytest.mark.parametrize("f", [0.0, 0.37])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_moments_of_amplitudes_that_are_no_numbers(f, bad):
    # as the formulas have it: x infinite gives NaN in g and, at F = 0, in the
    # logarithm (0 times infinity)
    torch, tn = require_cuda()
    k, n = 9001, 20
    a = _amps(k, n, 3)
    a[4321] = bad
    d = _dev(torch, a)
    with np.errstate(all="ignore"):
        ref = oxeb.pt_moments(oxeb.x_values(a, n), f)
    out = torch.empty(5, dtype=torch.float64, device="cuda")
    scratch = torch.empty(tn.tn_pt_moments_scratch_bytes(k), dtype=torch.uint8, device="cuda")
    tn.tn_pt_moments(d, k, n, f, out)
    got = [out.cpu().numpy()]
    tn.tn_pt_moments_scratch(d, k, n, f, out, scratch)
    for g in got + [out.cpu().numpy()]:
        assert np.array_equal(np.isnan(g), np.isnan(ref)) and np.array_equal(np.isinf(g), np.isinf(ref)), (g, ref)
    tn.tn_pt_moments_scratch(d, k, n, f, out, scratch, want_log=False)
    assert out[2].item() == 0.0
