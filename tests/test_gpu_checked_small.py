"""The bounds-checked build over the kernels that small systems and the FP64 path
run: one-cluster steps (lists built in the call, kept between calls, and taken over
from a forces call in sorted order) and FP64 forces and steps, alone and in a batch,
report no violation and give the normal build's bits."""
import os
import subprocess
import sys

import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import sys
import numpy as np
sys.path.insert(0, {root!r})
from paper_2010_01559_gb300 import build, capi
capi._lib = capi.load(build.build(check_bounds={checked}))
import torch
import paper_2010_01559_gb300 as rbe
from paper_2010_01559_gb300 import workloads
out = {{}}
e = workloads.electrolyte_1to1
for n, P in ((17, 1), (300, 10), (1000, 100), (3001, 10)):
    L = (n / 0.064) ** (1 / 3)
    wl = e(n, 0.064, 0.3 if L > 8 else 3.0, min(5.0, 0.45 * L), P, seed=n)
    h = rbe.RBE(rbe.params_from(wl.params, n_max=n))
    pos = torch.from_numpy(wl.pos_q()).cuda()
    vel = torch.zeros_like(pos)
    vel[:, :3] = torch.from_numpy(20.0 * wl.vel).cuda()
    step = torch.zeros(1, dtype=torch.int64, device="cuda")
    h.forces(pos, 0, energy=False)                 # the list in sorted order
    F = torch.zeros_like(pos)
    c0 = h.launch_count()
    for k in (1, 30, 3):
        h.step(pos, vel, k, step, F_out=F)
    assert h.launch_count() == c0 + 3              # one cluster each
    h.sync()
    assert h.list_stats()["builds"] >= 3
    p64, v64 = pos.double(), vel.double()
    F64, E64, phi = h.forces_f64(p64, 40, phi=True)
    h.step(p64, v64, 3, step)
    h.sync()
    for k, v in dict(F=F, pos=pos, F64=F64, E64=E64, phi=phi, p64=p64).items():
        out[k + str(n)] = v.cpu().numpy()
wls = [e(250, 0.064, u / 25.0, 5.0, 40, seed=3, stream=s) for s, u in enumerate((7.0, 30.0, 15.0))]
hb = rbe.RBEBatch([rbe.params_from(w.params) for w in wls], [w.n for w in wls])
xb = torch.from_numpy(np.concatenate([w.pos_q() for w in wls])).cuda().double()
Fb, _, _ = hb.forces_f64(xb, 2)
hb.sync()
out["Fb"] = Fb.cpu().numpy()
np.savez({path!r}, **out)
"""


def _run(checked, path):
    code = SCRIPT.format(root=ROOT, checked=checked, path=path)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    return np.load(path)


def test_no_violation_and_the_same_bits(tmp_path):
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    a, b = (_run(c, str(tmp_path / f"{c}.npz")) for c in (True, False))
    assert a.files == b.files
    for k in a.files:
        assert np.array_equal(a[k], b[k]), k
