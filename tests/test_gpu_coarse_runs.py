"""Coarsest inverses of a batch in which small operators (inverted on the host, a run of
neighbouring geometries copied at once) stand before, between and behind large ones (inverted on
the device): each geometry's solve takes about as many iterations as in a context of its own,
which it does not with another geometry's inverse (the coarsest correction is what makes the
iteration count independent of the size).  Bar: twice the largest count alone, since the batch
gives every geometry the same number of levels.
"""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


def channel(h, xlim, ylim):
    return w.channel_body(1 / h, ("circle", 0.5), Re=100.0, xlim=xlim, ylim=ylim)


def test_small_and_large_open_geometries(vip):
    small, large = channel(4, (-2, 3), (-1, 1)), channel(8, (-3, 9), (-3, 3))
    sets = [small, small, large, small, large, large, small]
    rng = np.random.default_rng(2)
    alone = {}
    for ns in (small, large):
        ctx = vip.solver_for(ns, set_state=False)
        b = rng.standard_normal(ns.n)
        alone[ns.n] = (b, *ctx.vip_solve("POISSON", b, np.zeros(ns.n), rtol=1e-10)[:2])
        ctx.close()
    assert len(alone) == 2
    ctx = vip.solver_for(sets, set_state=False)
    b = np.concatenate([alone[ns.n][0] for ns in sets])
    x, it, rr = ctx.vip_solve("POISSON", b, np.zeros(b.size), rtol=1e-10)
    ctx.close()
    assert rr <= 1e-10 and it <= 2 * max(a[2] for a in alone.values()), (it, [a[2] for a in alone.values()])
    o = 0
    for ns in sets:
        want = alone[ns.n][1]
        assert np.linalg.norm(x[o:o + ns.n] - want) <= 1e-6 * np.linalg.norm(want)
        o += ns.n
