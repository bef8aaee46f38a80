"""The network's kernels at the edges of their tiles: strips of exactly and just over 128 columns,
single rows and columns, CTAs whose range of tiles crosses from one strip to the next, and arrays
on the host, on the device and on the device at an odd address.

Same bars as test_gpu_cnn.py and for the same reasons: 2e-2 for the output against the FP64
network (BF16 storage), 1e-2 for gradients against the reference with BF16 at the same places.
The three kinds of arrays give the same bits.
"""
import ctypes as C

import numpy as np
import pytest

from oracle import cnn_oracle as co
from test_gpu_cnn import CH, bf16, bf16_reference_grads, ctx, eval_gpu, random_params, to_layers  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 128), (3, 129), (130, 3), (1, 640), (220, 700)])
def test_network_at_tile_edges(ctx, shape):  # noqa: F811
    import torch
    flat = random_params(ctx, 7)
    rng = np.random.default_rng(8)
    H, W = shape
    x = np.zeros((H, W, 16), np.float32)
    x[..., :6] = rng.standard_normal((H, W, 6))
    x = bf16(x)
    t = rng.standard_normal((H, W)).astype(np.float32)
    m = (rng.random((H, W)) > 0.2).astype(np.float32)
    y, g, loss = eval_gpu(ctx, x, t, m, flat.size)
    layers = to_layers(flat)
    ref = co.forward(layers, x.astype(np.float64))[0][..., 0]
    assert np.linalg.norm(y - ref) < 2e-2 * np.linalg.norm(ref)
    emu = bf16_reference_grads(layers, x.astype(np.float64), t.astype(np.float64), m.astype(np.float64))
    o = 0
    for k, (ci, cout) in enumerate(zip(CH[:-1], CH[1:])):
        n = 9 * ci * cout
        for got, want in ((g[o:o + n].reshape(emu[k][0].shape), emu[k][0]), (g[o + n:o + n + cout], emu[k][1])):
            assert np.linalg.norm(got - want) < 1e-2 * np.linalg.norm(want), (k, ci, cout)
        o += n + cout
    raw = torch.zeros(4 * x.size + 4, dtype=torch.uint8, device="cuda")
    raw[4:] = torch.from_numpy(x).cuda().reshape(-1).view(torch.uint8)
    td, md = torch.from_numpy(t).cuda(), torch.from_numpy(m).cuda()
    for xd in (torch.from_numpy(x).cuda(), raw[4:]):
        yd, gd, ld = torch.empty_like(td), torch.empty(flat.size, device="cuda"), C.c_double()
        ctx._check(ctx.L.vip_ws_eval(ctx.h, H, W, xd.data_ptr(), yd.data_ptr(), gd.data_ptr(), td.data_ptr(),
                                     md.data_ptr(), C.byref(ld)))
        assert np.array_equal(yd.cpu().numpy(), y) and np.array_equal(gd.cpu().numpy(), g) and ld.value == loss
