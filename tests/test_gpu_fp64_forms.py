"""The FP64 Fourier part in each pairing of its forms (phase tables or a sine and a
cosine per pair, for the structure factors and the force apart), at sizes on both sides
of where the tables stop paying, alone and in a batch: against plain 64-bit torch.

1e-12 relative RMS, the FP64 path's bound (phases of |k.r| up to some 1e3 turns)."""
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


def _system(n, alpha, P, seed):
    L = (n / 0.064) ** (1 / 3)
    rng = np.random.default_rng(seed)
    x = np.concatenate([rng.uniform(0, L, (n, 3)), rng.choice([-1.0, 1.0], (n, 1))], 1)
    return workloads.SystemParams(box=L, alpha=alpha, r_c=5.0, P=P, seed=seed, lj_eps=0.0), x


def _reference(torch, p, x, m, H):
    """Fourier force and its dE/dq of wave vectors m (sampling normalisation H)."""
    L = p.box
    k = m.double() * (2 * math.pi / L)
    coef = (H ** 3 - 1) / p.P * 4 * math.pi / (L ** 3 * (k * k).sum(1))
    t = (x[:, :3] / L) @ m.double().T
    t = 2 * math.pi * (t - torch.round(t))
    c, s = torch.cos(t), torch.sin(t)
    re, im = x[:, 3] @ c, x[:, 3] @ s
    F = -x[:, 3:] * ((c * (coef * im) - s * (coef * re)) @ k)
    return F, c @ (coef * re) + s @ (coef * im)


def _rel(a, b):
    return ((a - b).norm() / b.norm()).item()


@pytest.mark.parametrize("n,alpha,P", [
    (1000, 10.0, 5), (20000, 0.3, 10), (20000, 0.3, 33), (20000, 3.0, 10), (20000, 3.0, 129),
    (140000, 0.3, 20), (140001, 0.3, 200)])
def test_against_torch(rbe, n, alpha, P):
    import torch
    p, x = _system(n, alpha, P, 7)
    h = rbe.RBE(rbe.params_from(p, n_max=n))
    pos = torch.from_numpy(x).cuda()
    F, _, phi = h.forces_f64(pos, 4, parts=rbe.RBE_PART_FOURIER, energy=False, phi=True)
    h.sync()
    m = h.sample_k(4)[:, :3]
    rF, rphi = _reference(torch, p, pos, m, h.info().H)
    q = pos[:, 3]
    rphi = rphi - 2 * math.sqrt(alpha / math.pi) * q - math.pi / (p.box ** 3 * alpha) * q.sum()
    assert _rel(F[:, :3], rF) <= 1e-12 and _rel(phi, rphi) <= 1e-12
    h.close()


def test_batch_of_systems_where_tables_do_not_pay(rbe):
    import torch
    systems = [_system(n, a, P, 3 + i) for i, (n, a, P) in
               enumerate(((30000, 1.0, 7), (5000, 3.0, 12), (60000, 0.5, 3)))]
    h = rbe.RBEBatch([rbe.params_from(p) for p, _ in systems], [len(x) for _, x in systems])
    pos = torch.from_numpy(np.concatenate([x for _, x in systems])).cuda()
    F, _, _ = h.forces_f64(pos, 4, parts=rbe.RBE_PART_FOURIER, energy=False)
    m = h.sample_k(4)[:, :3]
    h.sync()
    off = k0 = 0
    for i, (p, x) in enumerate(systems):
        xi = torch.from_numpy(x).cuda()
        rF, _ = _reference(torch, p, xi, m[k0:k0 + p.P], h.info(i).H)
        assert _rel(F[off:off + len(x), :3], rF) <= 1e-12
        off, k0 = off + len(x), k0 + p.P
    h.close()
