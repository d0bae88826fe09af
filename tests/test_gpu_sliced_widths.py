"""The bit-sliced amplitude and chain kernels at the edges of their ranges: widths around a table
chunk (6 qubits) and a word (32, 62, 64), batches around a string word (32) and a block
(1024), term counts that leave partial tiles, against the string-per-thread kernel (the
allocation-free entry point: the same tile sums, so equal bits) and, for the chains, against the
amplitudes of the strings they end at and the one-step passes (equal bits)."""
import numpy as np
import pytest
import torch

from paper_1808_00128_gb300 import lrstab, workloads
from tests._gpu import require_cuda

pytestmark = pytest.mark.gpu


def _circuit(n, seed):
    """Clifford+T circuit whose terms have from none to many constraints, with a projector."""
    ops = workloads.random_clifford_t(n, 6 * n + 4, 3, seed)
    ops = [("H", q) for q in range(0, n, 2)] + ops
    if n >= 3:
        ops.insert(len(ops) // 2, ("CCZ", 0, 1, n - 1))
    return ops


def _sim(n, chi, seed):
    low = lrstab.lower_circuit(n, _circuit(n, seed))
    sim = lrstab.Simulator(n, 0)
    sim.init_terms(low, chi, mode="sparsify", seed=seed)
    sim.apply_clifford(low.gates)
    return sim


@pytest.mark.parametrize("n", [1, 2, 5, 6, 7, 12, 13, 31, 32, 33, 36, 37, 54, 60, 61, 62, 63, 64])
def test_sliced_amplitudes_equal_the_string_kernel(n):
    require_cuda()
    for chi, batches in ((7, (1, 1025)), (300, (31, 32, 33)), (2500, (64, 65, 513, 2049))):
        with _sim(n, chi, 70 + n) as sim:
            for b in batches:
                x = workloads.random_bitstrings(n, b, seed=b + n)
                x[: b // 2] = sim.sample_terms(b, seed=3).cpu().numpy().view(np.uint64)[: b // 2]
                x = torch.from_numpy(x.view(np.int64)).cuda()
                want = torch.empty((b, 2), dtype=torch.float64, device="cuda")
                sim.amplitude_noalloc(x, want)
                err = torch.empty(b, dtype=torch.float32, device="cuda")
                assert torch.equal(sim.amplitude(x), want), (n, chi, b)
                assert torch.equal(sim.amplitude(x, err=err), want), (n, chi, b)
                assert bool((err >= 0).all())


@pytest.mark.parametrize("n", [2, 6, 31, 33, 47, 62])
def test_chains_end_at_their_amplitudes(n):
    require_cuda()
    for chi, chains in ((5, 1), (700, 37), (8500, 130)):
        with _sim(n, chi, 40 + n) as sim:
            x0 = sim.sample_terms(chains, seed=9)
            ends = []
            for look in (2, 1):
                sim.set_tuning("mc_lookahead", look)
                sim.chains_init(x0)
                trace = torch.empty((7, chains), dtype=torch.int64, device="cuda")
                sim.metropolis(7, seed=4, trace=trace)
                xo = torch.empty(chains, dtype=torch.int64, device="cuda")
                po = torch.empty(chains, dtype=torch.float64, device="cuda")
                sim.metropolis(18, seed=4, step0=7, x_out=xo, p_out=po)
                ends.append((trace, xo, po))
            for a, b in zip(*ends):
                assert torch.equal(a, b), (n, chi)
            amp = torch.empty((chains, 2), dtype=torch.float64, device="cuda")
            sim.amplitude_noalloc(xo, amp)
            p = (amp ** 2).sum(1)
            assert torch.all((p - po).abs() <= 1e-5 * torch.clamp(p, min=2.0 ** -n)), (n, chi)
