"""Row pointers and candidate lists about the most counts that one block sums (16384): K = 2 n^2 candidate
counts below and above it, J = (n + 1)^2 row counts at it and above."""
import numpy as np
import pytest

from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [90, 91, 127, 128])   # K = 16200, 16562; J = 16384, 16641
def test_scan_threshold(n):
    from paper_2005_10775_gb300 import nlfem as nl
    m = I.split_square_mesh(0.0, float(n), n)
    ctx = nl.nl_create(0)
    try:
        keep = nl._Keep()
        D = nl.nl_assemble(ctx, nl.make_mesh(m, keep), nl.make_config(keep, 0.5, "barycenter", "dunavant7", "dunavant7",
                                                                      "const", 1.0, prec="fp64"))
        rp, ci, va = nl.nl_csr_download(ctx, D)
        nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    rows = np.repeat(np.arange(m.nv, dtype=np.int64), np.diff(rp))
    assert rp[0] == 0 and rp[-1] == ci.size
    assert (np.diff(ci)[np.diff(rows) == 0] > 0).all()   # sorted, distinct
    # a uniform grid: the rows of the nodes three lines from the boundary have the same columns relative to the
    # node (as line and column offsets)
    i, j = rows % (n + 1), rows // (n + 1)
    inner = (np.minimum(i, j) >= 3) & (np.maximum(i, j) <= n - 3)
    off = (ci // (n + 1) - j) * 1000 + (ci % (n + 1) - i)
    per = np.diff(rp)[np.unique(rows[inner])]
    assert (per == per[0]).all()
    assert (off[inner].reshape(-1, per[0]) == off[inner][:per[0]]).all()
    # the pattern is symmetric, and a constant lies in the kernel of D
    assert np.array_equal(np.sort(ci.astype(np.int64) * m.nv + rows), rows * m.nv + ci)
    assert np.abs(np.add.reduceat(va, rp[:-1])).max() <= 1e-13 * np.abs(va).max()
