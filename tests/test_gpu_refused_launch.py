"""A launch that CUDA refuses is reported by the call that made it, whatever
other runtime calls succeed after it: the direct FP64 structure factors of a batch of
2^23 wave vectors need 65536 rows of blocks, one more than a grid has."""
import pytest

from gpu_util import need_gpu, oracle_eval, rel_rms
from paper_2010_01559_gb300 import capi, workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbe():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_01559_gb300 as rbe
    return rbe


@pytest.mark.parametrize("graph", [False, True])
def test_refused_launch_is_reported(rbe, graph):
    import torch
    p = workloads.SystemParams(box=200.0, alpha=10.0, r_c=5.0, P=1 << 23, lj_eps=0.0)
    h = rbe.RBE(rbe.params_from(p, n_max=2))
    assert h.info().M > 560                      # the direct form
    h.set_graph(graph)
    pos = torch.tensor([[1.0, 2, 3, 1], [4, 5, 6, -1]], dtype=torch.float64, device="cuda")
    vel, step = torch.zeros_like(pos), torch.zeros(1, dtype=torch.int64, device="cuda")
    for call in (lambda: h.forces_f64(pos, 0), lambda: h.step(pos, vel, 2, step)):
        with pytest.raises(rbe.RBEError) as e:
            call()
        assert e.value.status == capi.RBE_ERR_CUDA
    h.sync()                                     # nothing is left behind
    h.close()
    wl = workloads.electrolyte_1to1(300, 0.064, 0.3, 5.0, 20, seed=2)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    F, _, _ = h.forces_f64(torch.from_numpy(wl.pos_q()).cuda().double(), 1)
    h.sync()
    assert rel_rms(F[:, :3].cpu().numpy(), oracle_eval(wl, 1)["F"]) <= 1e-12
    h.close()
