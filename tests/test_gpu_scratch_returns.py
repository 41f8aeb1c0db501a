"""A gradient that needs the memory of the second CTA's scratch per SM gives it
back: later batches run two CTAs per SM again."""

import numpy as np
import pytest

import paper_2605_29514_gb300 as stn
from workloads import D3_EXACT, theta_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_gradient_under_memory_pressure_keeps_the_scratch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    stn.build()
    w = D3_EXACT.with_(rounds=1, theta=0.1)
    records = 32  # whose states take more than the scratch of one CTA per SM
    sim = stn.Simulator(w, max_shots=2 * torch.cuda.get_device_properties(0).multi_processor_count)
    theta = theta_table(w, sim.n_pairs)
    rec = sim.sample_shots(records, 0, theta, stats=False)["records"]
    want = sim.logprob_grad(rec, theta)
    chi = [min(64, 2 ** min(k, 17 - k)) for k in range(18)]
    rotations = int(np.sum(stn.compile_program(w)[1][:, 0] == 6))  # op kind 6
    states = 16 * records * rotations * sum(2 * chi[k] * chi[k + 1] for k in range(17))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    room = int(states / 0.8 * 0.95)  # the states' share of the free memory is just too small
    filler = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
    before = torch.cuda.mem_get_info()[0]
    assert states > 0.8 * before
    got = sim.logprob_grad(rec, theta)
    after = torch.cuda.mem_get_info()[0]
    del filler
    torch.cuda.empty_cache()
    assert np.array_equal(got[0], want[0]) and np.allclose(got[1], want[1], rtol=1e-12, atol=0)
    assert abs(after - before) < 2 ** 26
    sim.close()
