"""Truncations with cutoffs at and below rounding, where every value counts: a
matrix that is short of full rank has no vector beyond its rank to keep."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn
from oracle.shot import make_program, run_shot
from workloads import D3_EXACT, theta_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("cutoff", [0.0, 1e-300, 1e-16, 1e-14])
@pytest.mark.parametrize("basis,theta,cap", [("Z", 0.05, 32), ("X", 0.1, 5)])
def test_cutoffs_at_rounding(precision, cutoff, basis, theta, cap):
    """Born probabilities against the oracle at the same cutoff: 1e-9 in
    complex128 and 5e-5 in complex64, the bounds of ordinary cutoffs."""
    w = D3_EXACT.with_(rounds=1, p=0.0, theta=theta, memory_basis=basis, precision=precision, chi_cap=cap,
                       svd_cutoff=cutoff, degeneracy_tol=1e-4)
    sim = stn.Simulator(w, max_shots=3)
    angles = theta_table(w, sim.n_pairs)
    out = sim.sample_shots(3, 5, angles)
    sim.close()
    prog = make_program(w)
    for s in range(3):
        ref = run_shot(w, 5 + s, angles, prog)
        assert list(out["bits"][s]) == list(ref.record)
        rb = np.array(ref.born)
        assert (np.abs(out["born"][s] - rb) / np.maximum(rb, 1e-4)).max() < (1e-9 if precision == 0 else 5e-5)
