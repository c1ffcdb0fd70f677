"""The FP64 path's kernels at the sizes where their tiles end: particle counts
around the 8-particle tables and the 16-lane groups, batches around the 128
wave vectors of a tile, a neighbourhood that overflows the candidate list, and
a sampling table too wide for shared memory (the direct form).

Tolerance: 1e-12 relative RMS, the FP64 path's against the oracle everywhere
(phases of |k.r| up to ~1e3 turns carry ~1e-13)."""
import numpy as np
import pytest

from gpu_util import need_gpu, oracle_eval, rel_rms
from paper_2010_01559_gb300 import workloads

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def rbe():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_01559_gb300 as rbe
    return rbe


def _check(rbe, wl, split=0):
    import torch
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    if split:
        h.set_tuning(0, 0, split, 0, 0)
    pos = torch.from_numpy(wl.pos_q()).cuda().double()
    F, E, phi = h.forces_f64(pos, 5, phi=True)
    Fm, _, _ = h.forces_f64(pos, 5, energy=False, phi=False)     # the force-only kernels
    h.sync()
    ref = oracle_eval(wl, 5, want_phi=True)
    assert rel_rms(F[:, :3].cpu().numpy(), ref["F"]) <= TOL
    assert rel_rms(Fm[:, :3].cpu().numpy(), ref["F"]) <= TOL
    assert rel_rms(phi.cpu().numpy(), ref["phi"]) <= TOL
    e = E[0].cpu().numpy()
    assert abs(e[0] - ref["E"][0]) <= TOL * np.abs(ref["E"][1:]).sum()
    h.close()


@pytest.mark.parametrize("n,P", [(65, 1), (66, 127), (71, 128), (72, 129), (250, 257), (1031, 513)])
@pytest.mark.parametrize("split", [1, 3, 9])
def test_tile_edges(rbe, n, P, split):
    _check(rbe, workloads.electrolyte_1to1(n, 0.064, 0.3, min(5.0, (n / 0.064) ** (1 / 3) / 2), P,
                                           seed=n + P), split)


@pytest.mark.parametrize("split", [1, 3, 9])
def test_crowded_neighbourhood(rbe, split):
    """400 charges of a 4 x 4 x 4 corner among 600: more than the 96 listed
    candidates within the cutoff."""
    rng = np.random.default_rng(3)
    p = workloads.SystemParams(box=30.0, alpha=0.3, r_c=5.0, P=20, seed=3, lj_eps=0.0)
    pos = rng.uniform(0, 30.0, (600, 3))
    pos[:400] = rng.uniform(0, 4.0, (400, 3))
    q = np.where(np.arange(600) % 2 == 0, 1.0, -1.0).astype(np.float32)
    wl = workloads.Workload("crowded", p, pos.astype(np.float32), q,
                            np.zeros((600, 3), np.float32))
    _check(rbe, wl, split)


def test_wide_sampling_table_takes_the_direct_form(rbe):
    """alpha L^2 = 4e5: half width M above the 560 the tables hold."""
    wl = workloads.electrolyte_1to1(300, 300 / 200.0 ** 3, 10.0, 5.0, 30, seed=9)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    assert h.info().M > 560
    h.close()
    _check(rbe, wl)


@pytest.mark.parametrize("u", [7.9, 8.0, 8.1, 15.9, 16.0, 16.1, 30.0])
def test_pair_terms_where_the_polynomials_change(rbe, u):
    """alpha r_c^2 at the two polynomials' ends and beyond them, and one system
    beyond them in a batch, which takes the library functions for all."""
    import torch
    def wl_of(u, seed):
        return workloads.electrolyte_1to1(250, 0.064, u / 25.0, 5.0, 40, seed=seed)
    wl = wl_of(u, 3)
    pos = torch.from_numpy(wl.pos_q().astype(np.float64)).cuda()
    ref = oracle_eval(wl, 5, want_phi=True)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=wl.n))
    F, E, phi = h.forces_f64(pos, 5, phi=True)
    h.sync()
    assert rel_rms(F[:, :3].cpu().numpy(), ref["F"]) <= TOL
    assert rel_rms(phi.cpu().numpy(), ref["phi"]) <= TOL
    h.close()
    both = [wl, wl_of(30.0, 4)]
    hb = rbe.RBEBatch([rbe.params_from(w.params) for w in both], [w.n for w in both])
    posb = torch.from_numpy(np.concatenate([w.pos_q() for w in both]).astype(np.float64)).cuda()
    Fb, _, _ = hb.forces_f64(posb, 5)
    hb.sync()
    assert rel_rms(Fb[:250, :3].cpu().numpy(), ref["F"]) <= TOL
    hb.close()
