"""Calls whose device buffers cannot be allocated (lrs_debug_limit_alloc makes the
allocations fail on the host): they report it, and leave nothing behind that a later call would
run on."""
import pytest
import torch

from paper_1808_00128_gb300 import lrstab, workloads
from tests._gpu import require_cuda

pytestmark = pytest.mark.gpu

OOM, STATE = -2, -5


def _sim(n=40, chi=3000, seed=5):
    low = lrstab.lower_circuit(n, workloads.random_clifford_t(n, 8 * n, 12, seed))
    sim = lrstab.Simulator(n, 0)
    sim.init_terms(low, chi, mode="sparsify", seed=seed)
    sim.apply_clifford(low.gates)
    return sim


def _chains(sim, x0, steps=20):
    x, p = torch.empty_like(x0), torch.empty(x0.numel(), dtype=torch.float64, device="cuda")
    sim.chains_init(x0)
    sim.metropolis(steps, seed=8, x_out=x, p_out=p)
    return x, p


@pytest.mark.parametrize("first", [0, 96])
def test_no_steps_on_the_chains_of_a_failed_start(first):
    """lrs_chains_init without memory for more chains: no chains, neither the new nor the old
    ones (whose states went with the failed allocation); then a start that fits."""
    require_cuda()
    sim = _sim()
    x0 = sim.sample_terms(200, seed=2)
    want = _chains(sim, x0)
    sim.close()
    sim = _sim()
    if first:
        _chains(sim, x0[:first].contiguous())
    sim.debug_limit_alloc(1000)
    with pytest.raises(lrstab.LrsError) as e:
        sim.chains_init(x0)
    assert e.value.status == OOM
    with pytest.raises(lrstab.LrsError) as e:
        sim.metropolis(1, seed=8)
    assert e.value.status == STATE
    sim.debug_limit_alloc(0)
    got = _chains(sim, x0)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    sim.close()
