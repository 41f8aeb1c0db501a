"""Bonds that a CTA with half of an SM decomposes from global scratch (a bond at
the cap beside one of 32), at odd caps, where a CTA's scratch has to be aligned for
16-byte numbers, and with an arena that shrinks the span stacks."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn
from oracle.shot import make_program, run_shot
from workloads import D3_EXACT, D5_BENCH, theta_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()


def born_error(got, want):
    return (np.abs(got - want) / np.maximum(want, 1e-4)).max()


def d5_shots(cap, precision, arena=0):
    w = D5_BENCH.with_(rounds=2, p=1e-3, theta=0.1, chi_cap=cap, precision=precision)
    sim = stn.Simulator(w, max_shots=3, arena_cap_bytes=arena)  # every second CTA's scratch would be misaligned
    out = sim.sample_shots(3, 0, theta_table(w, sim.n_pairs))
    sim.close()
    return out


def test_d5_odd_cap_against_complex128():
    """Equal records and Born probabilities to the single-precision level of
    two d = 5 rounds, 5e-5."""
    got, want = d5_shots(55, 1), d5_shots(55, 0)
    assert got["max_chi"].max() == 55
    assert np.array_equal(got["records"], want["records"])
    assert born_error(got["born"], want["born"]) < 5e-5


def test_shrunk_arena_changes_no_bit():
    """Span stacks of 9/10 of the plan's, in an odd number of 8-byte elements."""
    cap, n = 63, 49
    chi = [min(cap, 2 ** min(k, n - k)) for k in range(n + 1)]
    need = sum(8 * chi[k] * chi[k + 1] for k in range(n)) + sum(4 * c * c for c in chi[1:n])
    full, shrunk = d5_shots(cap, 1), d5_shots(cap, 1, 8 * (need * 9 // 10 | 1))
    assert full["max_chi"].max() == cap
    assert np.array_equal(full["records"], shrunk["records"]) and np.array_equal(full["born"], shrunk["born"])


@pytest.mark.parametrize("cap", [49, 63])
def test_d3_odd_caps_against_oracle(cap):
    w = D3_EXACT.with_(rounds=1, p=0.0, theta=0.2, memory_basis="X", chi_cap=cap, precision=1, svd_cutoff=5e-6,
                       degeneracy_tol=5e-6)
    sim = stn.Simulator(w, max_shots=3)
    theta = theta_table(w, sim.n_pairs)
    out = sim.sample_shots(3, 7, theta)
    prog = make_program(w)
    for s in range(3):
        ref = run_shot(w, 7 + s, theta, prog)
        assert list(out["bits"][s]) == list(ref.record)
        assert born_error(out["born"][s], np.array(ref.born)) < 5e-5
    sim.close()
