"""vip_apply on device arrays (read and written in place) against the same call on host arrays
(staged): the same sums in the same order, so the same bits, for every operator, on a batch of
a closed and an open geometry, with a NaN in the field, in place and at an odd address."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

OPS = ["LAPLACE", "VIP_E", "VIP_W", "VIP_N", "VIP_S", "GX", "GY", "HELM_U", "HELM_V", "POISSON"]


@pytest.mark.parametrize("sets", ["closed, open", "open", "periodic, closed"])
def test_device_and_host_arrays_agree(vip, sets):
    import torch
    make = {"closed": lambda: w.cavity(21), "periodic": lambda: w.periodic_box(20),
            "open": lambda: w.channel_body(1 / 4, ("circle", 0.5), xlim=(-2, 3), ylim=(-2, 2))}
    nss = [make[s]() for s in sets.split(", ")]
    ctx = vip.solver_for(nss, set_state=False)
    n = sum(s.n for s in nss)
    closed = sum(1 for s in nss if not (s.kind == w.KIND_OUTLET).any())
    for op in OPS:
        m = n + (closed if op == "POISSON" else 0)
        x = np.random.default_rng(1).standard_normal(m)
        x[m // 3] = np.nan
        ref = np.full(m, 7.0)
        ctx.vip_apply(op, x, ref)
        xd = torch.from_numpy(x).cuda()
        y = torch.full_like(xd, 7.0)
        ctx.vip_apply(op, xd, y)
        assert np.array_equal(y.cpu().numpy(), ref, equal_nan=True), op
        assert np.isnan(ref).any() and not np.isnan(ref).all()
        ctx.vip_apply(op, xd, xd)                       # in place
        assert np.array_equal(xd.cpu().numpy(), ref, equal_nan=True), op
        raw = torch.zeros(8 * m + 4, dtype=torch.uint8, device="cuda")
        raw[4:] = torch.from_numpy(x).cuda().view(torch.uint8)
        y.fill_(7.0)
        ctx.vip_apply(op, raw[4:], y)                   # not aligned as doubles
        assert np.array_equal(y.cpu().numpy(), ref, equal_nan=True), op
        one = torch.zeros(m, dtype=torch.float64, device="cuda")
        ctx.vip_apply(op, x, one)                       # host to device
        assert np.array_equal(one.cpu().numpy(), ref, equal_nan=True), op
    ctx.close()
