"""The FP64 path in the caller's length units: a system in reduced units and the
same one with every length times 2^-30 (near a nanometre in metres) and 2^20 give
the same energies, forces (times 1 / scale), potentials and steps.

The scaling is by powers of two, so that only the order of operations the code
takes with lengths rounds differently: 1e-12 relative RMS, the FP64 path's bound."""
import dataclasses

import numpy as np
import pytest

from gpu_util import need_gpu, rel_rms
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


def _scaled(p, s):
    """The system's parameters with lengths times s (energies and times as they are)."""
    return dataclasses.replace(p, box=p.box * s, alpha=p.alpha / s ** 2, r_c=p.r_c * s,
                               lj_sigma=p.lj_sigma * s, lj_rcut=p.lj_rcut * s,
                               coulomb_prefactor=p.coulomb_prefactor * s, mass=p.mass / s ** 2,
                               gamma=p.gamma / s ** 2)


@pytest.mark.parametrize("u", [7.5, 15.0, 30.0])
@pytest.mark.parametrize("scale", [2.0 ** -30, 2.0 ** 20])
def test_forces_energy_potential_and_steps(rbe, u, scale):
    import torch
    wl = workloads.electrolyte_1to1(400, 0.064, u / 25.0, 5.0, 60, seed=17)
    out = []
    for s in (1.0, scale):
        h = rbe.RBE(rbe.params_from(_scaled(wl.params, s), n_max=wl.n))
        pos = torch.from_numpy(wl.pos_q().astype(np.float64)).cuda()
        pos[:, :3] *= s
        vel = torch.zeros_like(pos)
        vel[:, :3] = torch.from_numpy(wl.vel.astype(np.float64) * s).cuda()
        F, E, phi = h.forces_f64(pos, 5, phi=True)
        Fm, _, _ = h.forces_f64(pos, 5, energy=False)
        step = torch.zeros(1, dtype=torch.int64, device="cuda")
        h.step(pos, vel, 5, step)
        h.sync()
        out.append([x.cpu().numpy() for x in (F * s, Fm * s, phi, E, pos[:, :3] / s,
                                              vel[:, :3] / s)])
        h.close()
    for name, a, b in zip(("F", "F alone", "phi", "E", "pos", "vel"), *out):
        assert np.isfinite(b).all(), name
        assert rel_rms(b, a) <= TOL, (name, rel_rms(b, a))
