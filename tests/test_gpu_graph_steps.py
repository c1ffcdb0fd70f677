"""Replayed MD steps of systems that the one-cluster kernel does not take (N = 4001
and an odd 12007, a batch, a handle without a list): the mixed path's graphs of one and
of several steps give the bits of plain launches, across calls of any length, from the
device counter and on host arrays.  Launch counts show that each side ran the separate
kernels, and that replays were graphs of whole steps."""
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


def _systems(kind):
    e = workloads.electrolyte_1to1
    if kind == "batch":
        return [e(n, 0.064, 0.3, 5.0, 40, seed=n, stream=i) for i, n in enumerate((500, 3000, 1777))]
    n, P, thermostat = {"langevin": (4001, 60, 0), "nose_hoover": (12007, 30, 2),
                        "no list": (4001, 60, 1)}[kind]
    kw = {1: dict(andersen_nu=5.0), 2: dict(nh_tau=0.5)}.get(thermostat, {})
    wl = e(n, 0.064, 0.3, 5.0, P, seed=n, thermostat=thermostat, **kw)
    if kind == "no list":
        wl.params.skin = -1.0
    return [wl]


def _handle(rbe, wls, graph):
    ps = [rbe.params_from(w.params, n_max=w.n) for w in wls]
    h = rbe.RBE(ps[0]) if len(wls) == 1 else rbe.RBEBatch(ps, [w.n for w in wls])
    h.set_graph(graph)
    return h


def _state(wls, torch):
    pos = torch.from_numpy(np.concatenate([w.pos_q() for w in wls])).cuda()
    vel = torch.zeros_like(pos)
    vel[:, :3] = torch.from_numpy(6.0 * np.concatenate([w.vel for w in wls])).cuda()
    return pos, vel, torch.zeros(1, dtype=torch.int64, device="cuda")


@pytest.mark.parametrize("kind", ["langevin", "nose_hoover", "no list", "batch"])
def test_replays_equal_plain_launches(rbe, kind):
    import torch
    wls = _systems(kind)
    n = 96
    h = _handle(rbe, wls, False)
    ref = _state(wls, torch)
    F0 = torch.zeros_like(ref[0])
    c0 = h.launch_count()
    h.step(*ref[:2], n, ref[2], F_out=F0)
    h.sync()
    per_step = (h.launch_count() - c0) / n
    assert per_step >= 4 and per_step == int(per_step)      # separate kernels
    # one call (96 >= 64 steps: graphs of eight at once); calls of 10 (one step at a
    # time first, then eight and the rest); of 1; and plain and replayed calls in turn
    for lengths in ([n], [10] * 9 + [6], [1] * n, [7, 64, 3, 22]):
        hg = _handle(rbe, wls, True)
        pos, vel, step = _state(wls, torch)
        F = torch.zeros_like(pos)
        c0 = hg.launch_count()
        for i, k in enumerate(lengths):
            if len(lengths) == 4:
                hg.set_graph(i % 2 == 1)
            hg.step(pos, vel, k, step, F_out=F)
        hg.sync()
        assert hg.launch_count() - c0 == per_step * n, lengths
        assert step.item() == n
        assert torch.equal(pos, ref[0]) and torch.equal(vel, ref[1]) and torch.equal(F, F0), lengths
        hg.close()
    # host arrays, page-locked and pageable
    for pinned in (True, False):
        hg = _handle(rbe, wls, True)
        p, v, _ = (t.cpu() for t in _state(wls, torch))
        if pinned:
            p, v = p.pin_memory(), v.pin_memory()
        done = 0
        for k in (1, 2, 5, 64, 24):
            hg.step_host(p, v, k, done)
            done += k
        assert torch.equal(p, ref[0].cpu()) and torch.equal(v, ref[1].cpu()), pinned
        hg.close()
    h.close()
