"""Handles of different sizes used by host threads of one process, each thread with its own:
the calls of one must not change what another's launches may use.  The threads' work is issued
on the same stream, so results are those of the same calls made alone, bit for bit.
"""
import ctypes as C
import threading

import numpy as np
import pytest

import workloads as w
from test_gpu_coarse_inverse import harness, lattice  # noqa: F401

pytestmark = pytest.mark.gpu


def run_together(*jobs):
    """Each job in a thread of its own, all started together; their results, or the first error."""
    out, start = [None] * len(jobs), threading.Barrier(len(jobs))

    def go(k):
        start.wait()
        try:
            out[k] = jobs[k]()
        except Exception as e:  # noqa: BLE001
            out[k] = e

    threads = [threading.Thread(target=go, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for r in out:
        if isinstance(r, Exception):
            raise r
    return out


def steps3d(vip, n, steps):
    ns = w.box3d(n, periodic=True, length=2 * np.pi)
    b = vip.build3d_for(ns)
    b.vip_3d_set_flow(10.0, 0.02, 1e-8, 1000)
    b.vip_3d_set_state(np.sin(ns.z), np.sin(ns.x), np.sin(ns.y), np.zeros(ns.n))
    for _ in range(steps):
        b.vip_3d_step(1)
    s = b.vip_3d_get_state()
    b.close()
    return s


def test_steps_of_small_and_large_3d_sets(vip):
    work = [(8, 400), (40, 200), (8, 400)]
    alone = [steps3d(vip, *k) for k in work]
    for a, b in zip(alone, run_together(*[lambda k=k: steps3d(vip, *k) for k in work])):
        assert all(np.array_equal(p, q) for p, q in zip(a, b))


def inverse(harness, coef, nbr, nx, ny, count):
    m = nx * ny
    pad = -m % 32
    coef = np.ascontiguousarray(np.pad(coef, ((0, 0), (0, pad))))
    nbr = np.ascontiguousarray(np.pad(nbr, ((0, 0), (0, pad)), constant_values=-1)).astype(np.int32)
    inv, inv32 = np.empty(m * m), np.empty(m * m, np.float32)
    one = [np.array([k], t) for k, t in ((nx, np.int32), (ny, np.int32), (0, np.int64))]
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)  # noqa: E731
    for _ in range(count):
        st = harness.run(1, C.c_int64(m + pad), *map(ptr, one), ptr(coef), ptr(nbr), C.c_int64(m * m), ptr(inv), ptr(inv32))
        if st != 0:
            raise RuntimeError(f"status {st}")
    return inv


def test_small_and_large_coarsest_operators(harness):
    """The set-up of contexts: coarsest operators whose substitution takes 16 and 64 KB of
    shared memory (a short lattice, and one that is periodic along y)."""
    work = [(9, 8, 0, 300), (40, 40, 1, 60), (9, 8, 0, 300)]
    args = [(*lattice(nx, ny, 0, py, True, np.random.default_rng(11)), nx, ny, c) for nx, ny, py, c in work]
    alone = [inverse(harness, *a[:4], 1) for a in args]
    got = run_together(*[lambda a=a: inverse(harness, *a) for a in args])
    assert all(np.array_equal(p, q) for p, q in zip(alone, got))
