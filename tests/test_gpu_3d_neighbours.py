"""Neighbour lists of the 3D build where its FP32 test of distances cannot decide, or only in
part: distances equal to rho, coordinates far from the origin, sizes whose squares leave FP32's
range, periodic boxes of one, two and three cells a side.  Lists are compared entry by entry with
the oracle's FP64 test (exact: both round step by step), at the nodes and at the VIPs above them."""
import dataclasses

import numpy as np
import pytest

import workloads as w
from oracle import vip_oracle3d as o3

pytestmark = pytest.mark.gpu


def moved(ns, d):
    return dataclasses.replace(ns, x=ns.x + d, y=ns.y - d, z=ns.z + 0.5 * d)


def scaled(ns, f):
    return dataclasses.replace(ns, x=ns.x * f, y=ns.y * f, z=ns.z * f, h=ns.h * f)


CASES = {
    "ties": (lambda: w.box3d(8), 3.0),
    "at 1e3": (lambda: moved(w.box3d(8, jitter=0.3), 1e3), 2.2),
    "at 1e6": (lambda: moved(w.box3d(8, jitter=0.3), 1e6), 2.2),
    "huge": (lambda: w.box3d(8, jitter=0.3, length=1e25), 2.2),
    "tiny": (lambda: scaled(w.box3d(8, jitter=0.3), 1e-21), 2.2),   # (box3d itself: absolute tolerances)
    "periodic 3": (lambda: w.box3d(7, periodic=True, jitter=0.3), 2.2),
    "periodic 2": (lambda: w.box3d(5, periodic=True, jitter=0.2), 2.2),
    "periodic ties": (lambda: w.box3d(8, periodic=True), 3.0),
    "periodic 4": (lambda: w.box3d(4, periodic=True, jitter=0.2), 2.2),
}


@pytest.mark.parametrize("name", CASES)
def test_neighbours_equal_the_oracles(vip, name):
    make, support = CASES[name]
    ns = make()
    b = vip.build3d_for(ns, support=support)
    pts, L, rho = np.stack([ns.x, ns.y, ns.z], 1), (ns.Lx, ns.Ly, ns.Lz), support * ns.h
    ptr, col, _ = b.vip_3d_get_stencil("NBR")
    rptr, ridx = o3.neighbours3(pts, rho, pts, L)
    assert np.array_equal(ptr, rptr) and np.array_equal(col, ridx)
    ii = np.nonzero(ns.kind == w.KIND_INTERIOR)[0]
    top = pts[ii].copy()
    top[:, 2] = top[:, 2] + 0.5 * ns.h[ii]
    rptr, ridx = o3.neighbours3(top, rho[ii], pts, L)
    ptr, col, _ = b.vip_3d_get_stencil("VIP_T")
    b.close()
    assert np.array_equal(np.diff(ptr)[ii], np.diff(rptr)) and np.array_equal(col, ridx)
