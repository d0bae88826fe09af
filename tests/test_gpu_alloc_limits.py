"""Calls whose device buffers cannot be allocated (lrs_debug_limit_alloc makes the
allocations fail on the host): they report it, and leave nothing behind that a later call would
run on."""
import numpy as np
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


@pytest.mark.parametrize("n", [7, 40, 64])
def test_amplitudes_without_memory_for_records(n):
    """lrs_amplitude when the records cannot be had: the string-per-thread kernel in the
    scratch of its sums, the same bits and bounds, nothing reallocated from call to call,
    and a capture that replays."""
    require_cuda()
    sim = _sim(n, 3000)
    x = sim.sample_terms(300, seed=4)
    out = torch.empty((300, 2), dtype=torch.float64, device="cuda")
    err = torch.empty(300, dtype=torch.float32, device="cuda")
    want, want_err = sim.amplitude(x, err=err).clone(), err.clone()
    sim.close()
    sim = _sim(n, 3000)
    sim.debug_limit_alloc(300 * 96 * 12 + 1024)      # 96 tiles: a sum and a bound each
    sim.amplitude(x, out=out, err=err)
    assert torch.equal(out, want) and torch.equal(err, want_err)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sim.amplitude(x, out=out)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    few, small = x[:50].contiguous(), torch.empty((50, 2), dtype=torch.float64, device="cuda")
    for _ in range(3):
        sim.amplitude(few, out=small)
        sim.amplitude(x, out=out, err=err)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    g.reset()
    sim.debug_limit_alloc(0)
    assert torch.equal(sim.amplitude(x), want)
    sim.close()


def test_amplitudes_with_room_for_some_records():
    """Scratch left by a norm estimate that holds some of the records: launches over parts of
    every tile, the same bits."""
    require_cuda()
    sim = _sim(40, 20000)
    x = sim.sample_terms(1500, seed=4)
    want = sim.amplitude(x).clone()
    sim.close()
    sim = _sim(40, 20000)
    sim.norm_estimate(4450, seed=1)                  # about 32.7 MB; 34.5 for all records
    sim.debug_limit_alloc(1000)
    assert torch.equal(sim.amplitude(x), want)
    sim.close()


def test_chain_counts_up_and_down_between_graph_replays():
    """Steps replayed from the context's graph (16 at a time) after the chains' buffers moved: the
    chains of a context that never held another number."""
    require_cuda()
    sim = _sim()
    x0 = sim.sample_terms(700, seed=2)
    want = {}
    for c in (100, 200, 700):
        one = _sim()
        want[c] = _chains(one, x0[:c].contiguous(), steps=33)
        one.close()
    for c in (100, 200, 100, 700, 100, 200, 700, 100):
        got = _chains(sim, x0[:c].contiguous(), steps=33)
        assert torch.equal(got[0], want[c][0]) and torch.equal(got[1], want[c][1]), c
    # new storage of the terms, and back
    low = lrstab.lower_circuit(40, workloads.random_clifford_t(40, 320, 12, 5))
    for chi in (9000, 3000):
        sim.init_terms(low, chi, mode="sparsify", seed=5)
        sim.apply_clifford(low.gates)
        got = _chains(sim, x0[:100].contiguous(), steps=33)
    assert torch.equal(got[0], want[100][0]) and torch.equal(got[1], want[100][1])
    sim.close()


@pytest.mark.parametrize("n", [40, 55])
def test_few_chains_without_memory_for_their_planes(n):
    """The steps of few chains whose planes cannot be had: the strings and, to the rounding of the
    sums, the probabilities of the chains that have them; through the calls of a sharded step
    and under capture too, nothing reallocated."""
    require_cuda()
    sim = _sim(n)
    x0 = sim.sample_terms(8, seed=2)

    def trace(steps, step0=0):
        tr = torch.empty((steps, 8), dtype=torch.int64, device="cuda")
        p = torch.empty(8, dtype=torch.float64, device="cuda")
        sim.metropolis(steps, seed=8, step0=step0, trace=tr, p_out=p)
        return tr, p

    sim.chains_init(x0)
    want, want_p = trace(40)
    assert int((want[-1] != x0).sum()) > 0
    sim.close()
    sim = _sim(n)
    sim.debug_limit_alloc(100_000)
    sim.chains_init(x0)
    a, _ = trace(15)
    row = torch.empty(8, dtype=torch.int64, device="cuda")
    for step in (15, 16):
        amp = sim.metropolis_propose(8, step)
        sim.metropolis_accept(amp, 8, step, trace=row)
        a = torch.cat([a, row[None]])
    b, p = trace(23, 17)
    assert torch.equal(torch.cat([a, b]), want)
    assert bool(((p - want_p).abs() <= 1e-5 * torch.clamp(want_p, min=2.0 ** -n)).all())
    with pytest.raises(lrstab.LrsError) as e:        # not for many
        sim.chains_init(sim.sample_terms(200, seed=2))
    assert e.value.status == OOM
    sim.chains_init(x0)
    x, p = torch.empty_like(x0), torch.empty_like(p)
    sim.metropolis(40, seed=8, x_out=x, p_out=p)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sim.chains_init(x0)
        sim.metropolis(40, seed=8, x_out=x, p_out=p)
    x.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(x, want[-1])
    g.reset()
    sim.close()


def test_learned_steps_of_chains_without_planes():
    require_cuda()
    n = 40
    net = lrstab.MLP(n, 64)
    net.set_params(dict(W1=np.zeros((64, n)), b1=np.zeros(64), W2=np.zeros((64, 64)), b2=np.zeros(64),
                        W3=np.zeros((n, 64)), b3=np.zeros(n)))
    out = []
    for limit in (0, 100_000):
        sim = _sim(n)
        x0 = sim.sample_terms(8, seed=2)
        sim.debug_limit_alloc(limit)
        sim.chains_init(x0)
        x = torch.empty_like(x0)
        lrstab.metropolis_learned(sim, net, 3, seed=4)
        sim.metropolis(9, seed=8, x_out=x)
        out.append(x)
        sim.close()
    net.close()
    assert torch.equal(*out)


@pytest.mark.parametrize("n", [9, 40, 63, 64])
def test_norm_estimate_in_fifteen_words_and_a_row_per_term(n):
    """Scratch of lrs_norm_estimate: the partial sums, n + 15 words a term and n + 2 a state."""
    require_cuda()
    sim = _sim(n, 100_000)
    want = sim.norm_estimate(96, seed=3).clone()
    sim.close()
    sim = _sim(n, 100_000)
    cap, tiles = 100_096, 1564                       # tiles of 64 terms
    sim.debug_limit_alloc((96 * tiles + 31) // 32 * 32 * 8 + 8 * (cap * (n + 15) + 96 * (n + 2)))
    assert torch.equal(sim.norm_estimate(96, seed=3), want)
    sim.close()
