"""What the scratch pool keeps mapped, measured as the device's free memory: bounded after a wait
and given back by the trim entry and by destroying a handle. The calls' outputs come from memory
that torch holds already, so every change of the free memory is the library's."""
import gc

import pytest
import torch

import paper_2502_02294_gb300 as dh

pytestmark = pytest.mark.gpu

MB = 1 << 20
KEEP = 512 * MB    # most the pool keeps after a wait
SLACK = 64 * MB    # granularity of the driver's mappings


def _x_adjoint(n):
    """A call function for the x adjoint at n^3 (20 n^3 floats of scratch), outputs cached by torch."""
    u = torch.ones(5, n, n, n, device="cuda")
    u[1:4] = 0.1
    lam = torch.ones_like(u)

    def call():
        dh.sweep_adjoint(u, lam, 0, 0.1)
        torch.cuda.synchronize()
    call()
    dh.scratch_trim()
    return call


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_a_large_call_keeps_no_more_than_the_bound():
    call = _x_adjoint(256)  # 1.34 GB of scratch
    before = _free()
    call()
    assert _free() >= before - KEEP - SLACK


def test_trim_gives_the_kept_memory_back():
    call = _x_adjoint(128)  # 168 MB of scratch
    before = _free()
    call()
    held = _free()
    assert held <= before - 100 * MB  # kept: the next call maps nothing
    dh.scratch_trim()
    assert _free() >= held + 100 * MB
    call()
    assert _free() <= before - 100 * MB


def test_destroying_a_handle_gives_the_kept_memory_back():
    call = _x_adjoint(128)
    sim = dh.Simulation(dh.default_params(n=16, box=16.0, n_steps=2, a_start=0.5, a_end=0.6))
    call()
    held = _free()
    sim.close()  # a 16^3 handle holds a few MB itself
    del sim
    gc.collect()
    assert _free() >= held + 100 * MB
