"""Handles of different sizes used by host threads of one process, each thread with its own:
the calls of one must not change what another's launches may use.  The threads' work is issued
on the same stream, so results are those of the same calls made alone, bit for bit.
"""
import threading

import numpy as np
import pytest

import workloads as w

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
