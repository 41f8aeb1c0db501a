"""Gradients whose backward states are cut at a tiny cap among equal Schmidt
values: a measurement taken back is a sum of branches of equal weight."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn
from workloads import D3_EXACT, theta_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cap", [1, 2, 3])
@pytest.mark.parametrize("basis,rule", [("Z", "adjacent_idle"), ("X", "adjacent_idle+diag_xx")])
def test_gradient_at_tiny_caps_is_finite(cap, basis, rule):
    """The kept branch overlaps the forward state, so a gradient exists.  In
    complex64, where the equal values are equal; in complex128 they differ in the
    last place, and which branch survives is rounding."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()
    w = D3_EXACT.with_(rounds=1, p=1e-3, theta=7e-7, theta_sign="random_pair", memory_basis=basis, pair_rule=rule,
                       chi_cap=cap, precision=1, svd_cutoff=1e-4, degeneracy_tol=0.0)
    sim = stn.Simulator(w, max_shots=5)
    theta = theta_table(w, sim.n_pairs)
    records = sim.sample_shots(5, 18, theta)["records"]
    logp, grad = sim.logprob_grad(records, theta, shot_offset=18)
    sim.close()
    assert np.all(np.isfinite(logp)) and np.all(np.isfinite(grad))
