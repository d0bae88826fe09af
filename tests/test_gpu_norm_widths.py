"""The bit-sliced norm kernel at the edges of its row counts: widths around its
register layouts (one and two matrix columns per lane, the stages of the elimination) and
terms from no free variable (|v| = 0) over the basis route to |v| = n, with L no multiple of the
32 states of a word.  Tolerance as in test_gpu_norm: 1e-5 max(eta, ||psi||^2)."""
import random

import numpy as np
import pytest

from paper_1808_00128_gb300 import lrstab
from tests._gpu import oracle_overlaps, oracle_terms, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 9, 10, 11, 16, 17, 32, 34, 40, 41, 48, 49, 52, 57, 64])
def test_eta_over_free_variables(n):
    require_cuda()
    rng = random.Random(900 + n)
    for hs in sorted({0, 1, min(n, 15), min(n, 16), min(n, 17), n // 2, n - 1, n}):
        # H on hs qubits, then CX / CZ / S mixing and two T gates: |v| = hs, with
        # constraints over all qubits and, through S and X = H S S H, nonzero constants
        ops = [("H", q) for q in range(n)] + [("Z", q) for q in range(0, n, 2)] + [("H", q) for q in range(n)]
        ops += [("H", q) for q in rng.sample(range(n), hs)]
        for _ in range(4 * n):
            a, b = rng.sample(range(n), 2)
            ops.append((rng.choice(["CX", "CZ"]), a, b))
            ops.append(("S", rng.randrange(n)))
        ops.insert(len(ops) - n, ("T", rng.randrange(n)))
        ops.insert(len(ops) - 2 * n, ("T", rng.randrange(n)))
        low = lrstab.lower_circuit(n, ops)
        with lrstab.Simulator(n, 0) as sim:
            sim.init_terms(low, 4, mode="exact")
            sim.apply_clifford(low.gates)
            L = 37
            eta = sim.norm_estimate(L, seed=n).cpu().numpy()
        terms, coefs, _ = oracle_terms(n, ops, 4, "exact")
        want = (2.0 ** n) * np.abs(oracle_overlaps(terms, coefs, n, n, L, parallel=n > 16)) ** 2
        assert np.all(np.abs(eta - want) <= 1e-5 * np.maximum(want, 1.0)), (n, hs)
