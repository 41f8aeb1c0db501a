"""An angle that is not finite reaches the device after the bonds have grown past
those that are decomposed in shared memory: the shot ends with a status, and the
context goes on."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn
from workloads import D3_EXACT, theta_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()


@pytest.mark.parametrize("precision,cap,cutoff", [(1, 64, 5e-6), (1, 256, 5e-6), (2, 256, 5e-6), (0, 256, 1e-12)])
def test_non_finite_bond_is_reported(precision, cap, cutoff):
    w = D3_EXACT.with_(rounds=2, p=0.0, theta=0.1, memory_basis="X", precision=precision, chi_cap=cap,
                       svd_cutoff=cutoff, degeneracy_tol=cutoff)
    sim = stn.Simulator(w, max_shots=2)
    theta = theta_table(w, sim.n_pairs)
    good = torch.tensor(theta, dtype=torch.float64, device="cuda")
    bad = torch.full_like(good, float("nan"))
    torch.cuda.synchronize()
    want = sim.sample_shots(2, 0, theta)
    sim.begin_batch(2, 0)
    for step in range(sim.n_steps):
        sim.apply_step_device(step, (bad if step == sim.n_steps - 1 else good).data_ptr())
    with pytest.raises(stn.StnError) as e:
        sim.read_records()
    assert e.value.status == stn.STN_ENUMERIC
    again = sim.sample_shots(2, 0, theta)
    assert np.array_equal(again["records"], want["records"]) and np.array_equal(again["born"], want["born"])
    sim.close()


@pytest.mark.parametrize("arena", [1, 4096, 16384, 65536])
@pytest.mark.parametrize("precision", [0, 1])
def test_arena_that_is_too_small_is_reported(precision, arena):
    """Sweeps that outgrow the span stacks at different points of the program."""
    w = D3_EXACT.with_(rounds=1, p=0.0, theta=0.1, memory_basis="X", precision=precision, svd_cutoff=5e-6,
                       degeneracy_tol=5e-6)
    sim = stn.Simulator(w, max_shots=200, arena_cap_bytes=arena)
    theta = theta_table(w, sim.n_pairs)
    with pytest.raises(stn.StnError) as e:
        sim.sample_shots(200, 0, theta)
    assert e.value.status == stn.STN_EOVERFLOW
    assert np.all(sim.sample_shots(200, 0, np.zeros_like(theta))["max_chi"] == 1) if arena > 4096 else True
    sim.close()
