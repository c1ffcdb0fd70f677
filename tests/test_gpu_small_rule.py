"""Which systems run as one cluster: those whose step is shorter that way, by particles,
wave vectors and neighbours (a water-like system with 500 neighbours is taken up to
some 900 charges only), whatever the tuning and the graphs."""
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


# density, r_c, n, P, one cluster
@pytest.mark.parametrize("density,r_c,n,P,one", [
    (0.064, 5.0, 1000, 100, True), (0.064, 5.0, 1000, 500, True), (0.064, 5.0, 3000, 10, True),
    (0.064, 5.0, 3000, 100, False), (0.064, 5.0, 2000, 200, False),
    (0.3, 4.0, 300, 10, True), (0.3, 4.0, 2000, 10, True), (0.3, 4.0, 2000, 100, False),
    (0.1, 10.0, 300, 100, True), (0.1, 10.0, 801, 50, True), (0.1, 10.0, 999, 10, False),
    (0.1, 10.0, 1200, 100, False), (0.5, 5.0, 1000, 50, False)])
def test_rule(rbe, density, r_c, n, P, one):
    import torch
    L = (n / density) ** (1 / 3)
    wl = workloads.electrolyte_1to1(n, density, 0.3, min(r_c, 0.45 * L), P, seed=n)
    for graph in (False, True):
        h = rbe.RBE(rbe.params_from(wl.params, n_max=n))
        h.set_graph(graph)
        h.set_tuning(64, 2, 0, 0, 2)
        pos = torch.from_numpy(wl.pos_q()).cuda()
        step = torch.zeros(1, dtype=torch.int64, device="cuda")
        c0 = h.launch_count()
        h.step(pos, torch.zeros_like(pos), 3, step)
        h.sync()
        assert (h.launch_count() - c0 == 1) == one
        h.close()
