"""vip_ws_eval on images of growing size on one context."""
import pytest
import torch

import workloads as w

pytestmark = pytest.mark.gpu


def evaluate(ctx, x, y):
    ctx._check(ctx.L.vip_ws_eval(ctx.h, x.shape[0], x.shape[1], x.data_ptr(), y.data_ptr(), None, None, None, None))


def test_memory_of_a_larger_image(vip):
    """A larger image grows the activations (six of 32 channels, two gradients of 32 and one of 16
    in BF16, two FP32 planes: 552 bytes a cell; allocations in steps of 2 MB) and nothing else."""
    ctx = vip.solver_for(w.cavity(24, Re=100.0), set_state=False)
    x, y = torch.zeros(1200, 1200, 16, device="cuda"), torch.empty(1200, 1200, device="cuda")
    evaluate(ctx, x[:32, :32].contiguous(), y)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    evaluate(ctx, x, y)
    assert before - torch.cuda.mem_get_info()[0] <= 552 * 1200 * 1200 + 11 * (2 << 20)
    ctx.close()
