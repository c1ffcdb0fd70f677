"""A system's FP64 results do not depend on the other systems of its batch: the same
bits beside a system whose alpha r_c^2 lies beyond the polynomial's range and beside
one within it."""
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


@pytest.mark.parametrize("u", [7.0, 15.0])
def test_results_do_not_depend_on_the_company(rbe, u):
    import torch
    def wl_of(u, seed):
        return workloads.electrolyte_1to1(250, 0.064, u / 25.0, 5.0, 40, seed=seed)
    wl = wl_of(u, 3)
    out = []
    for other in (7.0, 15.0, 30.0):
        both = [wl, wl_of(other, 4)]
        h = rbe.RBEBatch([rbe.params_from(w.params) for w in both], [w.n for w in both])
        pos = torch.from_numpy(np.concatenate([w.pos_q() for w in both]).astype(np.float64)).cuda()
        F, E, phi = h.forces_f64(pos, 5, phi=True)
        Fm, _, _ = h.forces_f64(pos, 5, energy=False)
        h.sync()
        out.append((F[:wl.n], Fm[:wl.n], E[0], phi[:wl.n]))
        h.close()
    for o in out[1:]:
        for a, b in zip(out[0], o):
            assert torch.equal(a, b)
