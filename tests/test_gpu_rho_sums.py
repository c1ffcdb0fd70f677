"""The mixed structure factors' sums: partial sums up to the fixed-point words' range."""
import numpy as np
import pytest

from gpu_util import need_gpu, rel_rms
from paper_2010_01559_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rbe():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    import paper_2010_01559_gb300 as rbe
    return rbe


def _handle(rbe, box, alpha, r_c, P, n):
    p = workloads.SystemParams(box=box, alpha=alpha, r_c=r_c, P=P, seed=2, lj_eps=0.0, skin=-1.0)
    return rbe.RBE(rbe.params_from(p, n_max=n))


@pytest.mark.parametrize("charge", [1000.0, 1200.0, -2000.0])
def test_partial_sums_up_to_the_range_of_the_words(rbe, charge):
    """Below 256 particles the words hold 2^-52 steps: a macroion of charge 1200 is
    a partial sum of 2^62.2 of them.  Against the FP64 path, the mixed path's 1e-5, on
    the other charges (the macroion's own term, 1e6 times theirs, leaves its rounding
    in the force on it)."""
    import torch
    rng = np.random.default_rng(4)
    h = _handle(rbe, 20.0, 0.3, 5.0, 40, 64)
    x = np.concatenate([rng.uniform(0, 20.0, (64, 3)), rng.choice([-1.0, 1.0], (64, 1))], 1)
    x[7, 3] = charge
    pos = torch.from_numpy(x.astype(np.float32)).cuda()
    F, E, _ = h.forces(pos, 3, parts=rbe.RBE_PART_FOURIER)
    Fm, _, _ = h.forces(pos, 3, parts=rbe.RBE_PART_FOURIER, energy=False)
    R, Er, _ = h.forces_f64(pos.double(), 3, parts=rbe.RBE_PART_FOURIER)
    h.sync()
    others = [i for i in range(64) if i != 7]
    for f in (F, Fm):
        assert rel_rms(f[others, :3].cpu().numpy(), R[others, :3].cpu().numpy()) <= 1e-5
    assert abs(E[0, 1].item() / Er[0, 1].item() - 1.0) <= 1e-5
    h.close()
