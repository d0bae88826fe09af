"""The scratch of lrs_amplitude: a captured call's buffers stay where they are while later calls
take no more strings, whatever their tile plans, and calls whose records take several launches
(every tile's sums continued from launch to launch) give the bits of one."""
import numpy as np
import pytest
import torch

from paper_1808_00128_gb300 import lrstab, workloads
from tests._gpu import require_cuda

pytestmark = pytest.mark.gpu


def _sim(n, chi, seed=6, circuit=None):
    ops = circuit or [("H", q) for q in range(0, n, 3)] + workloads.random_clifford_t(n, 6 * n, 8, seed)
    low = lrstab.lower_circuit(n, ops)
    sim = lrstab.Simulator(n, 0)
    sim.init_terms(low, chi, mode="sparsify", seed=seed)
    sim.apply_clifford(low.gates)
    return sim


def _strings(sim, count):
    x = workloads.random_bitstrings(sim.n, count, seed=count)
    x[::2] = sim.sample_terms(count, seed=3).cpu().numpy().view(np.uint64)[::2]
    return torch.from_numpy(x.view(np.int64)).cuda()


@pytest.mark.parametrize("n,chi,batch,fewer", [(50, 1 << 20, 4096, (1024, 700, 1)), (40, 1 << 16, 4097, (4096, 1024, 33))])
def test_fewer_strings_leave_a_captured_call_its_scratch(n, chi, batch, fewer):
    require_cuda()
    sim = _sim(n, chi)
    x = _strings(sim, batch)
    out = torch.empty((batch, 2), dtype=torch.float64, device="cuda")
    sim.amplitude(x, out=out)
    want = out.clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sim.amplitude(x, out=out)
    err = torch.empty(batch, dtype=torch.float32, device="cuda")
    small = torch.empty_like(out)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for b in fewer:
        sim.amplitude(x[:b].contiguous(), out=small[:b])
        sim.amplitude(x[:b].contiguous(), out=small[:b], err=err[:b])
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free   # nothing reallocated: the graph may be replayed
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    g.reset()
    sim.close()


@pytest.mark.parametrize("n,chi", [(62, 600001), (64, 1000000), (20, 2300000)])
def test_several_launches_equal_the_string_kernel(n, chi):
    """More terms than records: launches over parts of every tile, among them one that is
    empty for the last tile, against the allocation-free entry point (no records)."""
    require_cuda()
    sim = _sim(n, chi)
    for b in (1, 33, 100, 513, 1500):
        x = _strings(sim, b)
        want = torch.empty((b, 2), dtype=torch.float64, device="cuda")
        sim.amplitude_noalloc(x, want)
        err = torch.empty(b, dtype=torch.float32, device="cuda")
        assert torch.equal(sim.amplitude(x), want), b
        assert torch.equal(sim.amplitude(x, err=err), want), b
        mag = want.norm(dim=1)
        assert bool((err >= 0).all()) and bool((err[mag > 0] > 0).all())
    sim.close()


@pytest.mark.parametrize("n", [19, 31, 45, 53])
def test_capture_after_a_call_of_the_other_kind(n):
    """A call with bounds sizes the scratch for one without: the capture of the latter, whose
    kernel has then not run, and the other way round (at widths that no other test of this
    file runs)."""
    require_cuda()
    for bounds in (True, False):
        sim = _sim(n + bounds, 500)
        x = _strings(sim, 200)
        want, out = (torch.empty((200, 2), dtype=torch.float64, device="cuda") for _ in range(2))
        err = torch.empty(200, dtype=torch.float32, device="cuda")
        sim.amplitude(x, out=want, err=err if bounds else None)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            sim.amplitude(x, out=out, err=None if bounds else err)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        g.reset()
        sim.close()


@pytest.mark.parametrize("n", [6, 7, 31, 33, 50, 62, 64])
def test_blocks_of_several_tiles_equal_the_string_kernel(n):
    """Few strings of many terms: blocks of 16, 8 or 4 string words and two to eight tiles."""
    require_cuda()
    for chi in (20000, 77824):
        sim = _sim(n, chi)
        for b in (3, 33, 100, 300):
            x = _strings(sim, b)
            want = torch.empty((b, 2), dtype=torch.float64, device="cuda")
            sim.amplitude_noalloc(x, want)
            err = torch.empty(b, dtype=torch.float32, device="cuda")
            assert torch.equal(sim.amplitude(x), want), (chi, b)
            assert torch.equal(sim.amplitude(x, err=err), want), (chi, b)
        sim.close()
