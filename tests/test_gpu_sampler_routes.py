"""Both routes of lrs_mlp_sample (one launch of two, four or eight rows a block; a product per
bit) against the FP64 oracle: given the bits drawn, one forward pass of the oracle gives every
bit's probability, so each bit is checked with its uniform draw and each log q with the sum.
Tolerances as in test_gpu_mlp (a bit may differ within 1e-3 of its probability, log q within 5e-3)."""
import numpy as np
import pytest

from oracle import mlp as omlp
from oracle import rng as orng
from paper_1808_00128_gb300 import lrstab
from tests._gpu import require_cuda

pytestmark = pytest.mark.gpu


def _check(n, H, count):
    params = omlp.init_params(n, H, seed=n * H)
    net = lrstab.MLP(n, H)
    net.set_params(params)
    seed, s0 = 5, 300
    y, lq = net.sample(count, seed, s0)
    y, lq = y.cpu().numpy().view(np.uint64), lq.cpu().numpy()
    net.close()
    assert n == 64 or int(y.max()) < 1 << n
    rows = np.unique(np.concatenate([np.arange(min(count, 40)), np.arange(max(0, count - 40), count),
                                     np.random.default_rng(1).integers(0, count, 80)]))
    Y = omlp.bits_matrix(y[rows], n)
    logits, _ = omlp.forward(params, Y)
    p = 1 / (1 + np.exp(-logits))
    U = np.array([[orng.uniform(seed, (1 << 40) + s0 + int(r), i) for i in range(n)] for r in rows])
    wrong = (U < p) != (Y > 0)
    assert np.all(np.abs(U - p)[wrong] < 1e-3)
    assert wrong.sum() <= 3
    np.testing.assert_allclose(lq[rows], -omlp.nll(logits, Y), rtol=0, atol=5e-3)


# one launch: a count per number of rows a block (about 300 and 600 are the edges), units of one bit
# below and above a warp's two and a thread's one, widths below, at and above the 512 loaded ahead
@pytest.mark.parametrize("count", [1, 299, 305, 603, 611, 1100])
@pytest.mark.parametrize("n,H", [(5, 64), (12, 512), (3, 256), (33, 576), (64, 1024)])
def test_one_launch(n, H, count):
    require_cuda()
    _check(n, H, count)


# few qubits, wide layers, many samples: a product per bit; and the widest layers of one launch
@pytest.mark.parametrize("n,H,count", [(2, 4096, 64), (4, 1024, 3000), (10, 512, 8200), (30, 64, 20001), (20, 4096, 70),
                                       (20, 3200, 330), (50, 3264, 700)])
def test_wide_layers_and_many_samples(n, H, count):
    require_cuda()
    _check(n, H, count)
