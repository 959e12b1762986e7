"""Rows of a mesh whose triangles' sizes differ a thousandfold: the FP64 path's whole-triangle areas keep their
digits whatever the largest triangle of the mesh is.

Bar: 1e-12 of the row's own largest entry.  An entry is a sum of some hundred products of FP64 numbers, each
within a few roundings; areas rounded on a grid of the largest triangle would miss it by 1e-9 / 1e-12."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def two_scales(n, fine):
    """Split-square grid whose first n - 3 cells in each direction are `fine` wide, the last three 1/3."""
    m = I.split_square_mesh(0.0, 1.0, n)
    lines = np.concatenate([fine * np.arange(n - 2), fine * (n - 3) + np.arange(1, 4) / 3.0])
    vx = lines[np.rint(m.vx * n).astype(int)]
    vy = lines[np.rint(m.vy * n).astype(int)]
    return I.Mesh(vx=vx, vy=vy, tri=m.tri, node_in_omega=m.node_in_omega, elem_in_omega=m.elem_in_omega, h=m.h,
                  lo=m.lo, hi=m.hi, n=n)


@pytest.mark.parametrize("ball", ["barycenter", "overlap"])
def test_rows_of_small_triangles(ball):
    from paper_2005_10775_gb300 import nlfem as nl
    m, d = two_scales(16, 3e-4), 1e-3
    c = I.const_kernel_c(d)
    ref = O.to_csr(O.assemble(m, dict(delta=d, ball=ball, outer="dunavant7", inner="gauss4", kernel_c=c))).tocsr()
    ref.sort_indices()
    ctx = nl.nl_create(0)
    try:
        keep = nl._Keep()
        D = nl.nl_assemble(ctx, nl.make_mesh(m, keep),
                           nl.make_config(keep, d, ball, "dunavant7", "gauss4", "const", c, prec="fp64"))
        G = nl.to_scipy(ctx, D)
        nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    np.testing.assert_array_equal(G.indptr, ref.indptr)
    np.testing.assert_array_equal(G.indices, ref.indices)
    rows = np.repeat(np.arange(m.nv), np.diff(ref.indptr))
    top = np.zeros(m.nv)
    np.maximum.at(top, rows, np.abs(ref.data))
    err = np.zeros(m.nv)
    np.maximum.at(err, rows, np.abs(G.data - ref.data))
    assert (top > 0).all() and (err / top).max() <= 1e-12
