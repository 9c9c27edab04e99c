"""The scratch pool of the single-call entries: same results from several threads and streams,
bounded, given back with the last handle, and usable under graph capture."""
import threading

import pytest
import torch

import paper_2502_02294_gb300 as dh
from paper_2502_02294_gb300 import api

pytestmark = pytest.mark.gpu

KEEP = 512 << 20   # most the pool keeps between calls
SLACK = 64 << 20   # granularity of the driver's mappings


def _inputs(n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    u = torch.rand(5, n, n, n, device="cuda", generator=g)
    u[0] += 1.0
    u[1:4] -= 0.5
    u[4] += 2.0
    lam = torch.randn(5, n, n, n, device="cuda", generator=g)
    return u, lam


def test_threads_and_streams_get_their_own_scratch():
    cases = [(n, seed) for seed, n in enumerate((16, 33, 48, 64))]
    want = [api.sweep_adjoint(*_inputs(n, seed), 0, 0.1)[0] for n, seed in cases]
    data = [_inputs(n, seed) for n, seed in cases]
    torch.cuda.synchronize()
    got = [[] for _ in cases]

    def work(i):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for rep in range(20):
                got[i].append(api.sweep_adjoint(*data[i], 0, 0.1)[0])
                if rep % 3 == i % 3:
                    st.synchronize()
        st.synchronize()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(cases))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w, outs in zip(want, got):
        assert len(outs) == 20 and all(torch.equal(w, o) for o in outs)


def test_kept_memory_is_bounded_and_given_back():
    n = 256  # 20 n^3 floats: 1.34 GB of scratch, more than the pool keeps
    u, lam = _inputs(n, 0)
    api.sweep_adjoint(*_inputs(16, 0), 0, 0.1)
    sim = dh.Simulation(dh.default_params(n=16, box=16.0, n_steps=2, a_start=0.5, a_end=0.6))
    out = api.sweep_adjoint(u, lam, 0, 0.1)[0]
    del out
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    first = api.sweep_adjoint(u, lam, 0, 0.1)[0]
    torch.cuda.synchronize()
    again = api.sweep_adjoint(u, lam, 0, 0.1)[0]
    torch.cuda.synchronize()
    assert torch.equal(first, again)
    assert torch.cuda.mem_get_info()[0] >= free0 - KEEP - SLACK - 2 * first.numel() * 4
    api.sweep_adjoint(*_inputs(128, 1), 0, 0.1)
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0]
    del sim  # destroying a handle gives back what the pool holds
    import gc
    gc.collect()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= held


def test_capture_and_replay():
    n = 32
    u, lam = _inputs(n, 5)
    want = api.sweep_adjoint(u, lam, 0, 0.1)[0]
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = api.sweep_adjoint(u, lam, 0, 0.1)[0]
    for _ in range(2):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
