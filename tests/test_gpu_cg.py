"""nl_cg over row counts about its cooperative grid (16 rows a round and block, 16 rounds between the sums)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 305, 4863, 4865, 77825, 160001])
def test_row_counts_about_the_grid(n):
    # tridiag(-1, 9/4, -1): condition number below 17.  The residual recomputed on the host differs from the
    # solver's by a few roundings of |A||x| <= 4.25 * 4 |b|, below 1e-13 |b|
    from paper_2005_10775_gb300 import nlfem as nl
    i = np.arange(n)
    keep = np.stack([i > 0, i >= 0, i < n - 1], 1)
    cols = np.stack([i - 1, i, i + 1], 1)[keep].astype(np.int32)
    vals = np.tile([-1.0, 2.25, -1.0], (n, 1))[keep]
    rp = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64)
    dev = [torch.from_numpy(a).cuda() for a in (rp, cols, vals)]
    b = np.random.default_rng(n).normal(size=n)
    x = np.zeros(n)
    ctx = nl.nl_create(0)
    try:
        A = nl.nl_csr(n=n, nnz=len(vals), row_ptr=ctypes.c_void_p(dev[0].data_ptr()),
                      col_idx=ctypes.c_void_p(dev[1].data_ptr()), val=ctypes.c_void_p(dev[2].data_ptr()))
        try:
            torch.cuda.synchronize()
            nl.nl_cg(ctx, A, b, x, rtol=1e-11, max_it=1000)
        finally:   # the arrays are torch's
            A.row_ptr = A.col_idx = A.val = None
            nl.nl_csr_free(ctx, A)
    finally:
        nl.nl_destroy(ctx)
    res = b - 2.25 * x
    res[1:] += x[:-1]
    res[:-1] += x[1:]
    assert np.linalg.norm(res) <= (1e-11 + 1e-13) * np.linalg.norm(b)
