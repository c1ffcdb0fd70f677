"""A one-cluster MD step whose blocks do not hear from each other gives the call up:
RBE_ERR_TIMEOUT, with positions, velocities, friction and step index as before it,
a list that the next step builds anew, and correct steps afterwards.

In a process of its own with the bounds-checked build, which takes the wait limit from
the environment: 0 is one look at the barrier right after the block's own messages, so
that some block finds another's missing."""
import os
import subprocess
import sys

import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import copy, os, sys
sys.path[:0] = [{root!r}, os.path.join({root!r}, "tests")]
import numpy as np, torch
from paper_2010_01559_gb300 import build, capi
capi._lib = capi.load(build.build(check_bounds=True))
import paper_2010_01559_gb300 as rbe
from paper_2010_01559_gb300 import workloads
from gpu_util import oracle_eval, rel_rms

def gives_up(call):
    os.environ["RBE_TEST_CLUSTER_WAIT_NS"] = "0"
    try:
        call()
        return False
    except rbe.RBEError as e:
        return e.status == capi.RBE_ERR_TIMEOUT
    finally:
        del os.environ["RBE_TEST_CLUSTER_WAIT_NS"]

for n, P, thermostat in ((300, 10, 1), (1000, 100, 2), (17, 1, 0)):
    kw = {{1: dict(andersen_nu=20.0), 2: dict(nh_tau=0.3)}}.get(thermostat, {{}})
    L = (n / 0.064) ** (1 / 3)
    wl = workloads.electrolyte_1to1(n, 0.064, 0.3 if L > 8 else 3.0, min(5.0, 0.49 * L), P,
                                    seed=n, thermostat=thermostat, **kw)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=n))
    pos = torch.from_numpy(wl.pos_q()).cuda()
    vel = torch.zeros_like(pos)
    vel[:, :3] = torch.from_numpy(4.0 * wl.vel).cuda()
    step = torch.zeros(1, dtype=torch.int64, device="cuda")
    h.step(pos, vel, 6, step)
    h.sync()
    p0, v0, xi0, b0 = pos.clone(), vel.clone(), h.nose_hoover_xi(), h.list_stats()["builds"]

    def steps(k):
        h.step(pos, vel, k, step)
        h.sync()
    for k in (1, 6, 600):
        assert gives_up(lambda: steps(k)), (n, k)
        assert torch.equal(pos, p0) and torch.equal(vel, v0) and step.item() == 6
        assert h.nose_hoover_xi() == xi0
    hp, hv = p0.cpu().pin_memory(), v0.cpu().pin_memory()
    for k in (1, 600):
        assert gives_up(lambda: h.step_host(hp, hv, k, 6))
        assert torch.equal(hp, p0.cpu()) and torch.equal(hv, v0.cpu())
    F = torch.zeros_like(pos)
    h.step(pos, vel, 1, step, F_out=F)
    h.sync()
    assert step.item() == 7 and h.list_stats()["builds"] > b0
    w = copy.copy(wl)
    w.pos = p0[:, :3].cpu().numpy()
    assert rel_rms(F[:, :3].cpu().numpy(), oracle_eval(w, 6)["F"]) <= 1e-5
    if thermostat != 2:                      # (the friction has advanced)
        h.step_host(hp, hv, 1, 6)
        assert torch.equal(hp, pos.cpu()) and torch.equal(hv, vel.cpu())
    h.close()
print("ok")
"""


def test_a_call_whose_blocks_do_not_meet_is_given_up():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT)], capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    assert r.stdout.strip().splitlines()[-1] == "ok"
