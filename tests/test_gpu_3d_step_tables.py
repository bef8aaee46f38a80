"""The 3D step's sliced tables and its convection straight from the point lists: node counts
around whole slices of 32 rows, with and without wall rows, and supports whose lists are shorter
and longer than the 16 entries a warp copies at a time (up to 132 with a support of 3.1).

Both sides solve to a relative residual of 1e-13, so the fields agree to 1e-10 relative L2, the
bar of the 3D parity tests.  The tables hold what the step needs once: 7 points a node of 47
neighbours on average take 1.3 KB of indices and 4.9 KB of weights, the system 0.6 KB, three
differences of at most 94 entries 3.4 KB, the fields 0.3 KB: 10.5 KB a node.
"""
import numpy as np
import pytest
import torch

import workloads as w
from oracle import vip_oracle3d as o3

pytestmark = pytest.mark.gpu

CASES = {
    "cube6": (lambda: w.box3d(6, periodic=True, length=2 * np.pi, jitter=0.1, seed=3), 2.2),
    "cube8_support3.1": (lambda: w.box3d(8, periodic=True, length=2 * np.pi, jitter=0.2, seed=3), 3.1),
    "cube7_support1.75": (lambda: w.box3d(7, periodic=True, length=2 * np.pi), 1.75),
    "walls4": (lambda: w.box3d(4, jitter=0.2, seed=4), 2.2),
    "walls5": (lambda: w.box3d(5, jitter=0.2, seed=4), 2.5),
}


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("name", list(CASES))
def test_steps_match_oracle(vip, name):
    make, support = CASES[name]
    ns = make()
    Re, dt = 10.0, 0.01
    st = o3.abc_flow(ns.x, ns.y, ns.z, 0.0, Re)
    fs = o3.FractionalStep3(o3.Operators3(ns, support=support), Re, dt, rtol=1e-13)
    fs.set_state(*st)
    b = vip.build3d_for(ns, support=support)
    b.vip_3d_set_flow(Re, dt, 1e-13, 50000)
    b.vip_3d_set_state(*st)
    for _ in range(3):
        fs.step()
    b.vip_3d_step(3)
    for g, o, f in zip(b.vip_3d_get_state(), (fs.u, fs.v, fs.w, fs.p, fs.phi), ("u", "v", "w", "p", "phi")):
        assert rel(g, o) <= 1e-10, (f, rel(g, o))
    b.close()


def test_memory_of_a_stepping_handle(vip):
    ns = w.box3d(32, periodic=True, length=2 * np.pi)
    vip.build3d_for(ns).close()                       # the context's own memory
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    b = vip.build3d_for(ns)
    b.vip_3d_set_flow(10.0, 0.02, 1e-8, 1000)
    b.vip_3d_set_state(*o3.abc_flow(ns.x, ns.y, ns.z, 0.0, 10.0))
    b.vip_3d_step(1)
    used = before - torch.cuda.mem_get_info()[0]
    b.close()
    assert used <= 10500 * ns.n, used / ns.n
