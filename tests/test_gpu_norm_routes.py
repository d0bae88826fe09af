"""Routes of the norm kernel that small random cases do not take: a tile of terms per warp (large
calls) against tiles shared by a block's warps, whose bits are the same, and forms in which a
variable is joined to no other while many are left, whose rest is eliminated form by form."""
import random

import numpy as np
import pytest
import torch

from oracle import estimators as E
from paper_1808_00128_gb300 import lrstab, workloads
from tests._gpu import oracle_overlaps, oracle_terms, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 7, 12, 13, 20, 28, 31, 33, 37, 41, 45, 49, 52, 53, 57, 61, 64])
def test_tiles_of_a_warp_equal_tiles_of_a_block(n):
    """632 tiles: 288 states take them a warp each, 37 states a block each; eta_l is the same."""
    require_cuda()
    ops = [("H", q) for q in range(0, n, 2)] + workloads.random_clifford_t(n, 6 * n + 4, 5, 30 + n)
    if n >= 3:
        ops.insert(len(ops) // 2, ("CCZ", 0, 1, n - 1))
    low = lrstab.lower_circuit(n, ops)
    with lrstab.Simulator(n, 0) as sim:
        sim.init_terms(low, 20000, mode="sparsify", seed=n)
        sim.apply_clifford(low.gates)
        many, few = sim.norm_estimate(288, seed=9), sim.norm_estimate(37, seed=9)
        assert torch.equal(many[:37], few)
        assert bool(torch.isfinite(many).all()) and float(many.mean()) > 0


@pytest.mark.parametrize("n", [12, 20, 32, 33, 34, 40, 41, 48, 52, 56, 57, 60, 61, 64])
def test_forms_with_an_isolated_variable(n):
    """H on every qubit, then the CZ and S gates that cancel the rows of A_0 at some qubits: in
    state l = 0 of the group these variables are joined to no other, so that all its forms leave
    the sliced steps where the first of them is the pivot.  Tolerance as in test_gpu_norm."""
    require_cuda()
    seed, L = 77, 33
    A = E.draw_A(n, seed, 0)
    for alone in ([0], [2], [n // 2 & ~1, n - 1], [max(0, n - 12) & ~1], list(range(n))):
        ops = [("H", q) for q in range(n)]
        done = set()
        for p in alone:
            for q in range(n):
                if q != p and A[p][q] % 2 and (min(p, q), max(p, q)) not in done:
                    done.add((min(p, q), max(p, q)))
                    ops.append(("CZ", p, q))
            # diagonal 0 mod 4: S adds 3 to gamma, Z adds 2
            a = int(A[p][p]) % 4
            ops += {0: [], 1: [("S", p)], 2: [("Z", p)], 3: [("SDG", p)]}[a]
        rest = [q for q in range(n) if q not in alone]
        rng = random.Random(n)
        if rest:
            ops += [("T", rng.choice(rest)), ("T", rng.choice(rest))]
        low = lrstab.lower_circuit(n, ops)
        chi = low.exact_chi
        with lrstab.Simulator(n, 0) as sim:
            sim.init_terms(low, chi, mode="exact")
            sim.apply_clifford(low.gates)
            eta = sim.norm_estimate(L, seed=seed).cpu().numpy()
        terms, coefs, _ = oracle_terms(n, ops, chi, "exact")
        want = (2.0 ** n) * np.abs(oracle_overlaps(terms, coefs, n, seed, L, parallel=n > 16)) ** 2
        assert want[0] > 0 or rest            # the other variables may sum to zero in state 0
        assert np.count_nonzero(want) > L // 4
        assert np.all(np.abs(eta - want) <= 1e-5 * np.maximum(want, 1.0)), (n, alone)
