"""Host-array steps on page-locked arrays that the caller changes between calls (an
engine that rescales velocities, displaces particles or exchanges charges): every step
starts from what the arrays hold, at sizes whose velocities are read in place and
whose velocities are copied, with and without graphs."""
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


@pytest.mark.parametrize("n", [4001, 70001, 131071, 131073])
@pytest.mark.parametrize("graph", [False, True])
def test_steps_start_from_the_edited_arrays(rbe, n, graph):
    import torch
    wl = workloads.electrolyte_1to1(n, 0.064, 0.3, 5.0, 40, seed=11)
    h, d = (rbe.RBE(rbe.params_from(wl.params, n_max=n)) for _ in range(2))
    h.set_graph(graph)
    p, v = torch.from_numpy(wl.pos_q()).pin_memory(), torch.zeros((n, 4)).pin_memory()
    v[:, :3] = torch.from_numpy(wl.vel)
    for s in range(8):
        dp, dv = p.cuda(), v.cuda()
        h.step_host(p, v, 1, s)
        d.step(dp, dv, 1, torch.tensor([s], device="cuda"))
        d.sync()
        assert torch.equal(p, dp.cpu()) and torch.equal(v, dv.cpu()), s
        v[:, :3] *= -0.5 if s % 2 else 1.7
        p[s::97, :3] = (p[s::97, :3] + 0.01) % np.float32(wl.params.box)
        p[:, 3] = p[torch.randperm(n, generator=torch.Generator().manual_seed(s)), 3]
    h.close()
    d.close()
