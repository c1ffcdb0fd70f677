"""The mixed structure factors' sums: partial sums up to the fixed-point words' range,
and FP32 runs no longer than a named rho_chunk gives."""
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


@pytest.mark.parametrize("n,P,ulps,bound", [(50021, 137, 7, 1.5e-7), (140001, 128, 28, 5e-7)])
def test_fp32_runs_are_as_short_as_the_named_chunk(rbe, n, P, ulps, bound):
    """A clump at the origin (every phase 0, every cosine 1) of charges 1 + ulps 2^-23,
    which add up exactly in chains of up to 16 (64) terms but for 6e-8 (2.5e-7), and lose
    7/16 of a last place per term in chains twice as long: 4e-7 (1.5e-6) of the sum.
    The forces on probes, against those of charges 1 (exact sums), show that ratio."""
    import torch
    rng = np.random.default_rng(8)
    h = _handle(rbe, 60.0, 0.3, 5.0, P, n)
    x = np.zeros((n, 4), np.float32)
    x[:, 3] = 1.0
    x[-64:, :3] = rng.uniform(5.0, 55.0, (64, 3))
    v = 1.0 + ulps * 2.0 ** -23
    out = []
    for q in (1.0, v):
        x[:-64, 3] = q
        F, _, _ = h.forces(torch.from_numpy(x).cuda(), 3, parts=rbe.RBE_PART_FOURIER, energy=False)
        out.append(F[-64:, :3].double().cpu().numpy())
    h.sync()
    a, b = out
    ratio = (a * b).sum() / (a * a).sum()
    # (the probes' own share of rho, 64 of n charges at random phases, does not grow by v)
    assert abs(ratio / v - 1.0) <= bound, ratio / v - 1.0
    h.close()
