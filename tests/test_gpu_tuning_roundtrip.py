"""Passing the launch shapes in effect back to rbe_set_tuning leaves a handle as it
was: the same shapes and, to the last bit, the same forces on both paths."""
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


@pytest.mark.parametrize("n,P", [(8001, 50), (50021, 137), (140001, 100)])
def test_shapes_in_effect_can_be_set(rbe, n, P):
    import torch
    wl = workloads.electrolyte_1to1(n, 0.064, 0.3, 5.0, P, seed=3)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    pos = torch.from_numpy(wl.pos_q()).cuda()
    out = []
    for k in range(2):
        F, _, _ = h.forces(pos, 3, energy=False)
        Fe, E, _ = h.forces(pos, 3)
        F64, _, _ = h.forces_f64(pos.double(), 3, energy=False)
        h.sync()
        shapes = h.get_tuning()
        out.append((F, Fe, E, F64, torch.tensor(shapes)))
        h.set_tuning(*shapes)
    for a, b in zip(*out):
        assert torch.equal(a, b)
    h.close()
