"""The FP64 real-space pair terms to their own relative accuracy: isolated pairs up
to the cutoff, where erfc has fallen by seven orders, and pairs at the cutoff's edge
in a box a million cutoffs wide.

Bounds: a pair term's relative error is that of e^{-u} (u = alpha r^2, the
exponent's two roundings: 2 u 2^-53) and about ten more roundings, in the kernel and
in the reference alike: below 1e-13 for u <= 30."""
import math

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


def _pairs(box, spacing, side, dist, rng):
    """side^3 isolated pairs, one per site of a lattice; dist: their distances."""
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)
    a = (g + 0.5) * spacing
    d = rng.standard_normal(a.shape)
    d *= (dist / np.linalg.norm(d, axis=1))[:, None]
    pos = np.empty((2 * len(a), 3))
    pos[0::2], pos[1::2] = a, a + d
    assert pos.min() > 0 and pos.max() < box
    return pos


def _reference(pos, q, alpha):
    """Force on the first of each pair, phi of both, energy per pair (lB = 1)."""
    d = pos[1::2] - pos[0::2]
    F, phi, e = np.empty_like(d), np.empty(len(pos)), np.empty(len(d))
    sa = math.sqrt(alpha)
    for i, v in enumerate(d):
        r2 = float(v[0] * v[0] + v[1] * v[1] + v[2] * v[2])
        r = math.sqrt(r2)
        c = math.erfc(sa * r) / r
        g = c + 2.0 * sa / math.sqrt(math.pi) * math.exp(-alpha * r2)
        F[i] = -q[2 * i] * q[2 * i + 1] * g / r2 * v
        phi[2 * i], phi[2 * i + 1] = q[2 * i + 1] * c, q[2 * i] * c
        e[i] = q[2 * i] * q[2 * i + 1] * c
    return F, phi, e


def _check(rbe, box, alpha, r_c, pos, q):
    import torch
    p = workloads.SystemParams(box=box, alpha=alpha, r_c=r_c, P=10, seed=1, lj_eps=0.0)
    h = rbe.RBE(rbe.params_from(p, n_max=len(pos)))
    x = torch.from_numpy(np.concatenate([pos, q[:, None]], 1)).cuda()
    F, E, phi = h.forces_f64(x, 0, parts=rbe.RBE_PART_REAL, phi=True)
    Fm, _, _ = h.forces_f64(x, 0, parts=rbe.RBE_PART_REAL, energy=False)
    h.sync()
    rF, rphi, re = _reference(pos, q, alpha)
    for f in (F, Fm):
        f = f.cpu().numpy()[:, :3]
        for part, sign in ((f[0::2], 1.0), (f[1::2], -1.0)):
            rel = np.linalg.norm(part - sign * rF, axis=1) / np.linalg.norm(rF, axis=1)
            assert rel.max() <= 1e-13, rel.max()
    rel = np.abs(phi.cpu().numpy() / rphi - 1.0)
    assert rel.max() <= 1e-13, rel.max()
    assert abs(E[0, 2].item() - re.sum()) <= 1e-13 * np.abs(re).sum()
    h.close()


@pytest.mark.parametrize("u", [4.0, 7.9, 8.1, 15.9, 16.1, 30.0])
def test_relative_accuracy_up_to_the_cutoff(rbe, u):
    rng = np.random.default_rng(5)
    dist = 5.0 * np.linspace(0.9, 0.99999, 64)
    pos = _pairs(60.0, 15.0, 4, dist, rng)
    q = np.tile([1.0, 1.0, 1.0, -1.0], 32)
    q[::2] *= np.linspace(0.5, 2.0, 64)
    _check(rbe, 60.0, u / 25.0, 5.0, pos, q)


def test_cutoff_far_below_the_box(rbe):
    """L / r_c = 10^6: a unit of the 32-bit coordinates that preselect the pairs is
    2.3e-4 r_c, and no pair within the cutoff may be lost to it."""
    rng = np.random.default_rng(6)
    pos = _pairs(1e6, 1e5, 10, rng.uniform(0.999, 0.99999, 1000), rng)
    _check(rbe, 1e6, 1e-3, 1.0, pos, np.tile([1.0, -1.0], 1000))
