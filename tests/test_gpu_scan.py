"""Row pointers and candidate lists at the sizes where the one-block prefix sum changes course: below,
at and past a tile of 8192 counts, and past the largest array it takes (131072)."""
import numpy as np
import pytest

from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 63, 64, 65, 90, 257])
def test_row_pointers_and_pattern(n):
    from paper_2005_10775_gb300 import nlfem as nl
    # K = 2 n^2 counts of candidates (8, ..., 8192, ..., 132098), J = (n + 1)^2 row counts; a horizon of
    # half a cell keeps the lists short
    m = I.split_square_mesh(0.0, 1.0, n)
    ctx = nl.nl_create(0)
    try:
        keep = nl._Keep()
        D = nl.nl_assemble(ctx, nl.make_mesh(m, keep), nl.make_config(keep, 0.5 / n, "barycenter", "dunavant7",
                                                                      "dunavant7", "const", 1.0, prec="fp64"))
        rp, ci, va = nl.nl_csr_download(ctx, D)
        nnz = D.nnz
        nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    assert rp[0] == 0 and rp[-1] == nnz and (np.diff(rp) > 0).all()
    rows = np.repeat(np.arange(rp.size - 1), np.diff(rp))
    assert (np.diff(ci)[np.diff(rows) == 0] > 0).all()          # sorted, distinct columns in every row
    # the pattern is symmetric, and a constant lies in the kernel of D
    key = rows.astype(np.int64) * rp.size + ci
    assert np.array_equal(np.sort(ci.astype(np.int64) * rp.size + rows), key)
    sums = np.add.reduceat(va, rp[:-1])
    assert np.abs(sums).max() <= 1e-13 * np.abs(va).max()
