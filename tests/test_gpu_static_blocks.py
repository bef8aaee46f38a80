"""vip_bicgstab_static up to 512 rows, where the kernel goes on in one block if that block's shared
memory holds the matrix and in several otherwise: entry counts on both sides of the line (96 KB
less the row offsets for 128 rows), dense matrices of the smallest and largest counts with more
than one block, and a row offset array that does not start at 0.

Diagonally dominant matrices as in test_gpu_static_sizes.py: condition number below 10, so a
relative residual of 1e-12 leaves an error below 1e-11 (bar 1e-10).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LINE = ((96 << 10) - 129 * 8) // 12   # entries of 128 rows that just fit


@pytest.mark.parametrize("n,entries,shift", [(128, LINE, 0), (128, LINE + 1, 0), (65, 65 * 65, 0), (512, 512 * 512, 0),
                                             (512, 512 * 30, 0), (513, 513 * 40, 0), (300, 300 * 90, 7)])
def test_solves_in_one_block_or_several(vip, n, entries, shift):
    import torch
    rng = np.random.default_rng(n + entries)
    cnt = np.full(n, entries // n)
    cnt[:entries - cnt.sum()] += 1
    ptr = np.concatenate([[0], np.cumsum(cnt)]) + shift
    col, val = np.zeros(ptr[-1], np.int32), np.full(ptr[-1], np.nan)
    dense = np.zeros((n, n))
    for i in range(n):
        c = np.sort(np.append(rng.permutation(np.delete(np.arange(n), i))[:cnt[i] - 1], i))
        v = rng.uniform(-1.0, 1.0, c.size) * 2.0 / c.size
        v[c == i] = 4.0 + rng.random()
        col[ptr[i]:ptr[i + 1]], val[ptr[i]:ptr[i + 1]], dense[i, c] = c, v, v
    xs = rng.standard_normal(n)
    dev = [torch.from_numpy(a).cuda() for a in (ptr.astype(np.int64), col, val, dense @ xs)]
    out = []
    for _ in range(2):
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        st, it, rr = vip.vip_bicgstab_static(0, None, n, *dev, x, rtol=1e-12)
        assert st == vip.VIP_OK and rr <= 1e-11, (st, it, rr)
        out.append(x.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    assert np.linalg.norm(out[0] - xs) <= 1e-10 * np.linalg.norm(xs)
