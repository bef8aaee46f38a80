"""vip_bicgstab_static where its layout changes: one block, a few blocks, every SM; rows
whose part of the matrix fits a block's shared memory and rows too long for it; empty
rows' neighbours and ragged row lengths.

The matrices are diagonally dominant (4 + noise against off-diagonal sums below 2), so the
condition number is below 10 and a relative residual of 1e-12 leaves a relative error
below 1e-11 (bar 1e-10) against the solution the right-hand side was made from.
"""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,row", [(1, 0), (2, 1), (33, 3), (512, 5), (513, 5), (4097, 40), (20000, 7), (131071, 4),
                                   (131072, 31)])
def test_solves_at_the_edges_of_its_layout(vip, n, row):
    import torch
    rng = np.random.default_rng(n)
    cnt = rng.integers(0, row + 1, n)            # ragged rows, some with the diagonal only
    r = np.repeat(np.arange(n), cnt)
    c = rng.integers(0, n, r.size)
    v = rng.uniform(-1.0, 1.0, r.size) * 2.0 / max(row, 1)
    A = (sp.csr_matrix((v, (r, c)), shape=(n, n)) + sp.diags(4.0 + rng.random(n))).tocsr()
    A.sort_indices()
    xs = rng.standard_normal(n)
    b = A @ xs
    dev = [torch.from_numpy(a).cuda() for a in (A.indptr.astype(np.int64), A.indices.astype(np.int32), A.data, b)]
    out = []
    for _ in range(2):
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        st, it, rr = vip.vip_bicgstab_static(0, None, n, *dev, x, rtol=1e-12)
        assert st == vip.VIP_OK and rr <= 1e-11, (st, it, rr)
        out.append(x.cpu().numpy())
    assert np.array_equal(out[0], out[1])
    assert np.linalg.norm(out[0] - xs) <= 1e-10 * np.linalg.norm(xs)
    # the iteration limit is reported with the last iterate's residual
    if n > 512:
        x = torch.zeros(n, dtype=torch.float64, device="cuda")
        st, it, rr = vip.vip_bicgstab_static(0, None, n, *dev, x, rtol=1e-12, max_iters=1)
        assert st == vip.VIP_ERR_NOT_CONVERGED and it == 1 and rr > 1e-12
    # a zero right-hand side gives zero
    x = torch.ones(n, dtype=torch.float64, device="cuda")
    st, it, rr = vip.vip_bicgstab_static(0, None, n, *dev[:3], torch.zeros_like(dev[3]), x)
    assert st == vip.VIP_OK and it == 0 and rr == 0.0 and not x.any()
