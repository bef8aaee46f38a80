"""The 3D step's solve kernel on both sides of its memory rule: fewer slices than SMs, the
vectors and the table in a block's shared memory, the vectors alone, and neither (the three
velocity solves from about 167,000 rows on), with wall rows (long Neumann rows, in slices of
their own) and without.

Plane Poiseuille flow u = y (1 - y), p = -2x/Re in the walled unit cube is a fixed point of the
step; at a relative residual of 1e-11 it holds to 1e-9 (the bar of the 25^3 test).  The
exact ABC flow bounds the periodic step's error: 2.5e-4 in velocity at 32^3 after ten steps
of 0.02 (second order in space, so smaller on finer cubes).  A failed solve is reported and
the handle steps again after a new state.
"""
import numpy as np
import pytest

import workloads as w
from oracle import vip_oracle3d as o3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 31, 45, 58])
def test_poiseuille_is_a_fixed_point(vip, n):
    ns = w.box3d(n, jitter=0.25, seed=14)
    x, y, Re = ns.x, ns.y, 10.0
    u0 = y * (1 - y)
    b = vip.build3d_for(ns)
    b.vip_3d_set_flow(Re, 0.01, 1e-11, 50000)
    b.vip_3d_set_state(u0, 0 * u0, 0 * u0, -2 * x / Re)
    b.vip_3d_step(2)
    u, v, wv, p, _ = b.vip_3d_get_state()
    dp = p + 2 * x / Re
    drift = max(np.abs(u - u0).max(), np.abs(v).max(), np.abs(wv).max(), np.abs(dp - dp.mean()).max())
    steps, _, _, relres = b.vip_3d_get_iters()
    assert drift <= 1e-9 and steps == 2 and relres <= 1e-11, (drift, relres)
    b.close()


@pytest.mark.parametrize("n", [33, 60])
def test_abc_flow(vip, n):
    ns = w.box3d(n, periodic=True, length=2 * np.pi)
    Re, dt = 10.0, 0.02
    b = vip.build3d_for(ns)
    b.vip_3d_set_flow(Re, dt, 1e-10, 50000)
    b.vip_3d_set_state(*o3.abc_flow(ns.x, ns.y, ns.z, 0.0, Re))
    b.vip_3d_step(10)
    got = b.vip_3d_get_state()[:3]
    want = o3.abc_flow(ns.x, ns.y, ns.z, 10 * dt, Re)[:3]
    assert max(np.abs(g - e).max() for g, e in zip(got, want)) <= 2.5e-4
    b.close()


def test_failed_solve_is_reported(vip):
    ns = w.box3d(12, jitter=0.25, seed=13)
    u = np.where(np.isclose(ns.z, 1.0), 1.0, 0.0)
    z = np.zeros(ns.n)
    b = vip.build3d_for(ns)
    b.vip_3d_set_flow(100.0, 0.01, 1e-10, 3)
    b.vip_3d_set_state(u, z, z, z)
    with pytest.raises(vip.VipError) as e:
        b.vip_3d_step(1)
    assert e.value.status == vip.VIP_ERR_NOT_CONVERGED
    b.vip_3d_set_state(np.where(ns.kind == 0, np.nan, u), z, z, z)
    with pytest.raises(vip.VipError) as e:
        b.vip_3d_step(1)
    assert e.value.status == vip.VIP_ERR_NONFINITE
    b.vip_3d_set_flow(100.0, 0.01, 1e-10, 50000)
    b.vip_3d_set_state(u, z, z, z)
    b.vip_3d_step(1)
    assert b.vip_3d_get_iters()[3] <= 1e-10
    b.close()
