"""The matrix in any unit of length: the same mesh, horizon and polygon in metres, nanometres and far
smaller and larger units, against the FP64 oracle in the same unit.  FP32 holds neither products of areas
nor fourth powers of lengths in most of these units."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32c": 1e-6}   # the paths' stated accuracies, of max|D|


@pytest.fixture(scope="module")
def nl():
    from paper_2005_10775_gb300 import nlfem
    return nlfem


@pytest.fixture(scope="module")
def ctx(nl):
    c = nl.nl_create(0)
    yield c
    nl.nl_destroy(c)


@pytest.mark.parametrize("kernel,ball", [("const", "nocaps"), ("const", "approxcaps"), ("const", "exactcaps"),
                                         ("const", "ngon"), ("const", "barycenter"), ("inv_dist", "ngon")])
@pytest.mark.parametrize("unit", [1e-30, 1e-11, 1e-9, 1e6, 1e11])
@pytest.mark.parametrize("prec", ["fp64", "fp32c"])
def test_units_of_length(nl, ctx, unit, kernel, ball, prec):
    m = I.split_square_mesh(0.0, 1.0, 12, jitter=0.2, seed=3)
    d = 0.21 * unit
    m = dataclasses.replace(m, vx=m.vx * unit, vy=m.vy * unit)
    c = I.const_kernel_c(d) if kernel == "const" else I.inv_dist_kernel_c(d)
    off = I.ngon_offsets(32, d) if ball == "ngon" else None
    ref = O.assemble(m, dict(delta=d, ball=ball, outer="dunavant7", inner="dunavant7", kernel=kernel, kernel_c=c,
                             ngon_off=off), want_hash=True)
    keep = nl._Keep()
    mesh = nl.make_mesh(m, keep)
    cfg = nl.make_config(keep, d, ball, "dunavant7", "dunavant7", kernel, c, off, prec=prec)
    D = nl.nl_assemble(ctx, mesh, cfg)
    try:
        G = nl.to_scipy(ctx, D)
    finally:
        nl.nl_csr_free(ctx, D)
    R = O.to_csr(ref).tocsr()
    R.sort_indices()
    np.testing.assert_array_equal(G.indptr, R.indptr)
    np.testing.assert_array_equal(G.indices, R.indices)
    assert np.abs(G.data - R.data).max() <= TOL[prec] * np.abs(R.data).max()
    h, n, q = nl.nl_interactions(ctx, mesh, cfg)
    np.testing.assert_array_equal(n, ref["count_a"])
    np.testing.assert_array_equal(q, ref["qp_a"])
    np.testing.assert_array_equal(h, ref["hash_a"])
