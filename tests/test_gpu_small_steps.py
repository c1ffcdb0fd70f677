"""MD steps that run as one cluster, at the sizes where its shares end: ranks
without particles (fewer than 16, 17) or without wave vectors (P < 16), odd
shares, 32 to 4 lanes per particle, one cell (r_c > L/3); against the oracle,
against the separate kernels (which a profiled handle runs), and across calls.

Tolerances: the mixed path's 1e-5 relative RMS and the per-particle bound; after
12 steps at dt = 1e-3 the two paths' positions differ by a few FP32 roundings of
the box (1e-5 of it allowed)."""
import copy

import numpy as np
import pytest

from gpu_util import assert_per_particle, need_gpu, oracle_eval, rel_rms
from paper_2010_01559_gb300 import workloads

pytestmark = pytest.mark.gpu
SIZES = [(9, 3, 0), (16, 16, 1), (17, 1, 0), (33, 17, 2), (250, 5, 2), (300, 10, 1), (513, 33, 0),
         (1000, 100, 2), (1023, 129, 1), (1025, 100, 0), (2047, 64, 0), (3001, 10, 1),
         (700, 600, 0)]


@pytest.fixture(scope="module")
def rbe():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_01559_gb300 as rbe
    return rbe


def _workload(n, P, thermostat):
    L = (n / 0.064) ** (1 / 3)
    kw = {1: dict(andersen_nu=20.0), 2: dict(nh_tau=0.3)}.get(thermostat, {})
    alpha = 0.3 if L > 8 else 3.0               # keeps k = 0 rare in a tiny box
    return workloads.electrolyte_1to1(n, 0.064, alpha, min(5.0, 0.49 * L), P, seed=n,
                                      thermostat=thermostat, **kw)


def _state(wl, torch, scale=1.0):
    pos = torch.from_numpy(wl.pos_q()).cuda()
    vel = torch.zeros_like(pos)
    vel[:, :3] = torch.from_numpy(wl.vel * np.float32(scale)).cuda()
    return pos, vel, torch.zeros(1, dtype=torch.int64, device="cuda")


@pytest.mark.parametrize("n,P,thermostat", SIZES)
def test_against_oracle_and_separate_kernels(rbe, n, P, thermostat):
    import torch
    wl = _workload(n, P, thermostat)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    ref = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    ref.profile(True)                           # one launch per kernel
    a, b = _state(wl, torch, 6.0), _state(wl, torch, 6.0)
    c0 = h.launch_count()
    h.step(a[0], a[1], 11, a[2])
    assert h.launch_count() - c0 == 1           # the call was one launch
    before = a[0].clone()
    Fa, Fb = torch.zeros_like(a[0]), torch.zeros_like(b[0])
    h.step(a[0], a[1], 1, a[2], F_out=Fa)
    for _ in range(11):
        ref.step(b[0], b[1], 1, b[2])
    ref.step(b[0], b[1], 1, b[2], F_out=Fb)
    h.sync()
    ref.sync()
    w2 = copy.copy(wl)
    w2.pos = before[:, :3].cpu().numpy()
    o = oracle_eval(w2, 11)
    F = Fa[:, :3].cpu().numpy()
    assert rel_rms(F, o["F"]) <= 1e-5
    assert_per_particle(F, o["F"], (n, P))
    assert a[2].item() == b[2].item() == 12
    L = wl.params.box
    d = (a[0] - b[0])[:, :3].double()
    d -= L * torch.round(d / L)
    assert d.abs().max().item() <= 1e-5 * L
    assert (a[1] - b[1]).abs().max().item() <= 1e-3
    assert h.list_stats()["builds"] == ref.list_stats()["builds"]
    assert h.list_stats()["max_count"] == ref.list_stats()["max_count"]
    if thermostat == 2:
        assert abs(h.nose_hoover_xi()[0] - ref.nose_hoover_xi()[0]) <= 1e-4 * max(
            1.0, abs(ref.nose_hoover_xi()[0]))
    # a forces call goes over the list the cluster left
    b0 = h.list_stats()["builds"]
    Ff, _, _ = h.forces(before, 11, energy=False)
    assert h.list_stats()["builds"] == b0
    assert rel_rms(Ff[:, :3].cpu().numpy(), o["F"]) <= 1e-5
    h.close()
    ref.close()


@pytest.mark.parametrize("n,P,thermostat", [(300, 10, 1), (1000, 100, 2), (1023, 129, 0)])
def test_calls_of_any_length_are_bitwise_equal(rbe, n, P, thermostat):
    """40 steps in one call, in calls of 1, 3 and 13, and over a list that a
    forces call built: the same state to the last bit (but for the last one's
    first list, whose order is the sort's)."""
    import torch
    wl = _workload(n, P, thermostat)
    out = []
    for per in (40, 1, 3, 13):
        h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
        pos, vel, step = _state(wl, torch, 4.0)
        done = 0
        while done < 40:
            k = min(per, 40 - done)
            h.step(pos, vel, k, step)
            done += k
        h.sync()
        out.append((pos, vel, h.list_stats()["builds"]))
        h.close()
    for p, v, b in out[1:]:
        assert torch.equal(p, out[0][0]) and torch.equal(v, out[0][1]) and b == out[0][2]
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    pos, vel, step = _state(wl, torch, 4.0)
    h.forces(pos, 0, energy=False)              # builds the list in sorted order
    F = torch.zeros_like(pos)
    h.step(pos, vel, 1, step, F_out=F)
    assert h.list_stats()["builds"] == 1
    o = oracle_eval(wl, 0)
    assert rel_rms(F[:, :3].cpu().numpy(), o["F"]) <= 1e-5
    h.close()
