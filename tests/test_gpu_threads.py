"""Handles of different size used from several host threads at once: no call is
refused or disturbed by another handle's launches (kernel attributes belong to the
process, not to a handle), and every thread's trajectory is the one it gets alone."""
import ctypes
import threading

import numpy as np
import pytest

from gpu_util import need_gpu
from paper_2010_01559_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbe():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_01559_gb300 as rbe
    return rbe


def _run(rbe, torch, wl, calls, bits):
    """calls steps, one per call, straight through the C ABI (no Python between two
    calls but the loop, so that the threads' calls overlap)."""
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    pos = torch.from_numpy(wl.pos_q()).cuda()
    vel = torch.zeros_like(pos)
    vel[:, :3] = torch.from_numpy(wl.vel).cuda()
    if bits == 64:
        pos, vel = pos.double(), vel.double()
    step = torch.zeros(1, dtype=torch.int64, device="cuda")
    h.step(pos, vel, 1, step)
    call = h.lib.rbe_step_f64 if bits == 64 else h.lib.rbe_step
    args = (h.handle, wl.n, ctypes.c_void_p(pos.data_ptr()), ctypes.c_void_p(vel.data_ptr()), 1,
            ctypes.c_void_p(step.data_ptr()))
    refused = sum(call(*args) != 0 for _ in range(calls - 1))
    assert refused == 0, (wl.n, refused, h.lib.rbe_last_error(h.handle))
    h.sync()
    h.close()
    return pos, vel, step.item()


@pytest.mark.parametrize("bits,calls,sizes", [
    (32, 20000, ((1000, 100), (250, 10), (950, 90), (240, 8))),      # one-cluster steps
    (64, 2000, ((400, 40), (401, 41), (1000, 40))),                  # FP64 tables of M 30 .. 250
])
def test_handles_of_different_size_from_several_threads(rbe, bits, calls, sizes):
    import torch
    alpha = (0.3, 0.3, 0.3, 0.3) if bits == 32 else (15.0, 40.0, 0.3)
    wls = [workloads.electrolyte_1to1(n, 0.064, a, 5.0, P, seed=n)
           for (n, P), a in zip(sizes, alpha)]
    alone = [_run(rbe, torch, w, calls, bits) for w in wls]
    got, errors = [None] * len(wls), []

    def work(k):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                got[k] = _run(rbe, torch, wls[k], calls, bits)
        except Exception as e:                       # reported by the main thread
            errors.append((k, e))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(wls))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for a, b in zip(alone, got):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2] == b[2] == calls
