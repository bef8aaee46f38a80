"""The Krylov launch's work items, reductions and coarse-tile passes at the sizes where
their dispatch changes: a block with a few slices (several lanes per row), runs of four
slices that share a stencil next to single slices (channels), blocks that hold one, two or
more systems (batches of tiny cavities beside a large one), cells of more than four nodes
(curved boundaries).

Every form stops on its own FP64 residual, so the residual of the returned solution,
formed here by SciPy from the exported operator, meets the tolerance for every system up to
the rounding of one operator application (row of at most 32 entries: 1e-14 relative to
|A| |x|, taken as 1e-11 of |b| for these sizes' condition numbers below 1e5).  The same
call twice gives the same bits: the reductions' order is fixed.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import workloads as w

pytestmark = pytest.mark.gpu

RTOL = 1e-9
CASES = {
    "periodic16": lambda: [w.periodic_box(16)],
    "cavity9": lambda: [w.cavity(9, Re=100.0)],
    "cavity75": lambda: [w.cavity(75, Re=400.0)],
    "circle_h8": lambda: [w.channel_body(1 / 8, ("circle", 0.5), Re=100.0)],
    "circle_h13": lambda: [w.channel_body(1 / 13, ("circle", 0.5), Re=100.0)],
    "bumpy_h20": lambda: [w.channel_body(1 / 20, ("sines", 1.0, [(0.05, 12), (0.02, 31)]), Re=200.0)],
    "triangles2": lambda: [w.triangle_cavity(70, Re=200.0), w.triangle_cavity(41, Re=300.0)],
    "tiny_beside_large": lambda: [w.cavity(6, Re=100.0 + k) for k in range(60)] + [w.cavity(200, Re=400.0)],
}


@pytest.mark.parametrize("form", ["fp64", "mixed", "mg32"])
@pytest.mark.parametrize("name", list(CASES))
def test_solves_meet_the_tolerance_in_every_system(vip, name, form):
    nss = CASES[name]()
    ctx = vip.solver_for(nss, set_state=False)
    prec = {"fp64": vip.VIP_PREC_FP64, "mixed": vip.VIP_PREC_MIXED, "mg32": vip.VIP_PREC_MG32}[form]
    closed = [not (ns.kind == vip.VIP_NODE_OUTLET).any() for ns in nss]
    n = sum(ns.n for ns in nss)
    system = np.concatenate([np.full(ns.n, g) for g, ns in enumerate(nss)])
    for which in ("POISSON", "HELM_U"):
        ptr, col, val = ctx.vip_get_stencil(which)
        rows = ptr.size - 1
        A = sp.csr_matrix((val, col, ptr), shape=(rows, rows))
        sysrow = system
        if which == "POISSON":  # one extra row per closed geometry, in order
            sysrow = np.concatenate([system, [g for g, c in enumerate(closed) if c]]).astype(int)
            assert rows == n + sum(closed)
        b = np.random.default_rng(3).standard_normal(rows)
        out = []
        for _ in range(2):
            x, it, rr = ctx.vip_solve(which, b, np.zeros(rows), precision=prec, rtol=RTOL, max_iters=20000)
            assert rr <= RTOL and it > 0
            out.append(x)
        assert np.array_equal(out[0], out[1])
        r2 = np.bincount(sysrow, (b - A @ out[0]) ** 2)
        b2 = np.bincount(sysrow, b ** 2)
        assert np.sqrt((r2 / b2).max()) <= RTOL + 1e-11, (which, np.sqrt(r2 / b2).max())
    ctx.close()
