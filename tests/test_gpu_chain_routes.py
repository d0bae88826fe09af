"""Few chains and many: how many threads share a (chain, column) at the start, and how many
threads take the sums, depends on the size of the call; a chain's strings and probabilities
are the same bits whatever the others."""
import pytest
import torch

from paper_1808_00128_gb300 import lrstab, workloads
from tests._gpu import require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 12, 33, 40, 62])
def test_few_chains_equal_the_first_of_many(n):
    require_cuda()
    ops = [("H", q) for q in range(0, n, 2)] + workloads.random_clifford_t(n, 6 * n + 4, 6, 50 + n)
    if n >= 3:
        ops.insert(len(ops) // 2, ("CCZ", 0, 1, n - 1))
    low = lrstab.lower_circuit(n, ops)
    for chi in (60, 20000):
        with lrstab.Simulator(n, 0) as sim:
            sim.init_terms(low, chi, mode="sparsify", seed=n)
            sim.apply_clifford(low.gates)
            x0 = sim.sample_terms(1500, seed=5)
            for look in (2, 1):
                sim.set_tuning("mc_lookahead", look)
                ends = {}
                for c in (1500, 1, 8, 90):
                    x, p = torch.empty_like(x0[:c]), torch.empty(c, dtype=torch.float64, device="cuda")
                    tr = torch.empty((3, c), dtype=torch.int64, device="cuda")
                    sim.chains_init(x0[:c].contiguous())
                    sim.metropolis(3, seed=6, trace=tr)
                    sim.metropolis(17, seed=6, step0=3, x_out=x, p_out=p)
                    ends[c] = (tr, x, p)
                for c in (1, 8, 90):
                    many = [ends[1500][0][:, :c], ends[1500][1][:c], ends[1500][2][:c]]
                    # P at the start sums tiles of its own plan: equal once a move was accepted
                    moved = (many[0][-1] != x0[:c]) | (many[1] != x0[:c])
                    assert torch.equal(ends[c][0], many[0]) and torch.equal(ends[c][1], many[1]), (chi, c)
                    assert torch.equal(ends[c][2][moved], many[2][moved]), (chi, c)
                    assert torch.allclose(ends[c][2], many[2], rtol=1e-5, atol=1e-5 * 2.0 ** -n)
