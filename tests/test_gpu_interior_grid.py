"""The scatter's grid for interior pairs on a uniform mesh, where every pair rounds the same way: with a ball that
holds the whole mesh every block M_ab is |T_a| |T_b| c / 9, and entries whose nodes share no triangle are sums
of those alone.

Bar: a pair is at least 2^31 / 67.5 units of the grid (a ninth of an area product, where a row's bound is at most
7.5 areas and two roundings to powers of two below 2^30, and the grid is eight times finer), so it rounds by at
most 1.6e-8 of itself; on the rows' own grid it would be up to 1.26e-7."""
import numpy as np
import pytest

from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [13, 15, 16])   # 4.3e-8, 1.0e-7 and 6.0e-8 on the rows' grid
def test_interior_pairs_of_equal_triangles(n):
    from paper_2005_10775_gb300 import nlfem as nl
    m = I.split_square_mesh(0.0, 1.0, n)
    vals = {}
    ctx = nl.nl_create(0)
    try:
        for prec in ("fp64", "fp32c"):
            keep = nl._Keep()
            D = nl.nl_assemble(ctx, nl.make_mesh(m, keep),
                               nl.make_config(keep, 2.0, "barycenter", "gauss3", "gauss3", "const", 1.0, prec=prec))
            rp, ci, vals[prec] = nl.nl_csr_download(ctx, D)
            nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    rows = np.repeat(np.arange(m.nv), np.diff(rp))
    apart = np.maximum(np.abs(rows % (n + 1) - ci % (n + 1)), np.abs(rows // (n + 1) - ci // (n + 1))) > 1
    assert apart.sum() > 0.9 * ci.size   # every pair of nodes is an entry
    err = np.abs(vals["fp32c"] - vals["fp64"])[apart] / np.abs(vals["fp64"])[apart]
    assert err.max() <= 1.65e-8
