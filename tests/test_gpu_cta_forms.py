"""A shot's result does not depend on its batch: batches of more shots than SMs
run the round kernel compiled for two CTAs per SM, smaller ones the one that has
the registers of one."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn
from workloads import D3_EXACT, D5_BENCH, theta_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

C64 = dict(precision=1, svd_cutoff=5e-6, degeneracy_tol=5e-6)
WORKLOADS = {
    "d3_z": D3_EXACT.with_(rounds=1, p=0.02, **C64),
    "d3_x": D3_EXACT.with_(rounds=1, p=0.0, theta=0.0225, memory_basis="X", **C64),
    "d3_c128": D3_EXACT.with_(rounds=1, p=0.02),
    "d5_cap32": D5_BENCH.with_(rounds=1, theta=0.05, chi_cap=32),
}


@pytest.mark.parametrize("name", WORKLOADS)
def test_batch_size_changes_no_bit(name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()
    shots = torch.cuda.get_device_properties(0).multi_processor_count + 40
    sim = stn.Simulator(WORKLOADS[name], max_shots=shots)
    theta = theta_table(WORKLOADS[name], sim.n_pairs)
    large, small = sim.sample_shots(shots, 0, theta), sim.sample_shots(64, 0, theta)
    sim.close()
    for key in ("records", "born", "max_chi", "logp", "discarded"):
        assert np.array_equal(large[key][:64], small[key]), key
