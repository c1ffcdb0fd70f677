"""Host-buffer MD steps of a system larger than one cluster runs (N = 8001 and an
odd 20011): page-locked arrays, one and several steps per call, direct launches
and graph replay, and pageable arrays reproduce the device calls bit for bit,
over steps that build the list and steps that walk it."""
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


@pytest.mark.parametrize("n,thermostat", [(8001, 0), (20011, 2)])
def test_host_steps_equal_device_steps(rbe, n, thermostat):
    import torch
    kw = dict(nh_tau=0.5) if thermostat == 2 else {}
    wl = workloads.electrolyte_1to1(n, 0.064, 0.3, 5.0, 60, seed=11, thermostat=thermostat, **kw)

    def handle():
        return rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))

    v0 = np.zeros((wl.n, 4), np.float32)
    v0[:, :3] = 8.0 * wl.vel                     # rebuilds every few steps
    h = handle()
    pd, vd = torch.from_numpy(wl.pos_q()).cuda(), torch.from_numpy(v0.copy()).cuda()
    sd = torch.zeros(1, dtype=torch.int64, device="cuda")
    h.step(pd, vd, 24, sd)
    h.sync()
    assert h.list_stats()["builds"] >= 2
    for pinned in (True, False):
        for graph in (False, True):
            for per in (1, 2, 12):
                hh = handle()
                hh.set_graph(graph)
                p, v = torch.from_numpy(wl.pos_q().copy()), torch.from_numpy(v0.copy())
                if pinned:
                    p, v = p.pin_memory(), v.pin_memory()
                for s in range(0, 24, per):
                    hh.step_host(p, v, per, s)
                assert torch.equal(p, pd.cpu()) and torch.equal(v, vd.cpu()), (pinned, graph, per)
                hh.close()
    h.close()
