"""The mixed structure factors at the batches where a block's groups change (1 to
1025 wave vectors: 64 groups down to one, one to three tiles, 128 and 256 threads)
and at particle counts around a pass, with and without energies; and list steps at
the sizes where the sort and the build change form (16 lanes per particle or one,
one cluster or four kernels).

Tolerances: the mixed path's, 1e-5 relative RMS on forces and dE/dq and 1e-6 on the
energy; list against cell scan 1e-5 + 1e-6 |F| per particle (one missing pair moves
a force by 7e-5)."""
import copy

import numpy as np
import pytest

from gpu_util import energy_rel, need_gpu, oracle_eval, rel_rms
from paper_2010_01559_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbe():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_01559_gb300 as rbe
    return rbe


@pytest.mark.parametrize("P", [1, 2, 5, 16, 63, 65, 127, 128, 129, 170, 255, 257, 300, 511, 513,
                               700, 1025])
@pytest.mark.parametrize("n", [71, 1025])
def test_batch_sizes(rbe, P, n):
    import torch
    wl = workloads.electrolyte_1to1(n, 0.064, 0.3, min(5.0, 0.49 * (n / 0.064) ** (1 / 3)), P,
                                    seed=P)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    pos = torch.from_numpy(wl.pos_q()).cuda()
    ref = oracle_eval(wl, 7, want_phi=True)
    F, E, phi = h.forces(pos, 7, phi=True)
    Fn, _, _ = h.forces(pos, 7, energy=False)
    h.sync()
    assert rel_rms(F[:, :3].cpu().numpy(), ref["F"]) <= 1e-5
    assert rel_rms(Fn[:, :3].cpu().numpy(), ref["F"]) <= 1e-5
    assert rel_rms(phi.cpu().numpy(), ref["phi"]) <= 1e-5
    assert energy_rel(E[0].cpu().numpy(), ref["E"]) <= 1e-6
    h.close()


def test_batch_of_systems_with_different_batch_sizes(rbe):
    import torch
    e = workloads.electrolyte_1to1
    systems = [e(200 + 37 * i, 0.064, 0.3, 5.0, P, seed=40 + i, stream=i)
               for i, P in enumerate((1, 40, 130, 257, 513))]
    h = rbe.RBEBatch([rbe.params_from(w.params) for w in systems], [w.n for w in systems])
    pos = torch.from_numpy(np.concatenate([w.pos_q() for w in systems])).cuda()
    F, E, _ = h.forces(pos, 2)
    h.sync()
    off = 0
    for s, w in enumerate(systems):
        ref = oracle_eval(w, 2)
        assert rel_rms(F[off:off + w.n, :3].cpu().numpy(), ref["F"]) <= 1e-5
        assert energy_rel(E[s].cpu().numpy(), ref["E"]) <= 1e-6
        off += w.n
    h.close()


@pytest.mark.parametrize("n", [19455, 19457, 65536, 65537])
def test_list_steps_where_the_sort_and_the_build_change_form(rbe, n):
    import torch
    wl = workloads.electrolyte_1to1(n, 0.064, 0.3, 5.0, 20, seed=21)
    sp = copy.copy(wl.params)
    sp.skin = -1.0
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    hc = rbe.RBE(rbe.params_from(sp, n_max=wl.n))
    h.set_graph(True)
    pos = torch.from_numpy(wl.pos_q()).cuda()
    vel = torch.zeros_like(pos)
    vel[:, :3] = torch.from_numpy(20.0 * wl.vel).cuda()
    step = torch.zeros(1, dtype=torch.int64, device="cuda")
    F = torch.zeros_like(pos)
    for s in range(8):
        before = pos.clone()
        h.step(pos, vel, 1, step, F_out=F)
        Fc, _, _ = hc.forces(before, s, energy=False)
        dev = (F - Fc)[:, :3].double().norm(dim=1)
        bound = 1e-5 + 1e-6 * Fc[:, :3].double().norm(dim=1)
        assert bool((dev <= bound).all()), (s, float((dev / bound).max()))
    assert h.list_stats()["builds"] >= 2
    h.sync()
    h.close()
    hc.close()
