"""The singular kernel with a horizon below the triangles' size, where many triangles outside the disc pass the
tangent's empty test and an edge-distance test takes them out, and regions in the near field have caps: records
and pattern bit-exact with the FP64 oracle, values within the paths' stated accuracies."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32c": 1e-6}


@pytest.mark.parametrize("ball", ["ngon", "nocaps", "approxcaps", "exactcaps"])
@pytest.mark.parametrize("prec", ["fp64", "fp32c"])
def test_singular_small_horizon(ball, prec):
    from paper_2005_10775_gb300 import nlfem as nl
    d = 0.07
    m = I.split_square_mesh(0.0, 1.0, 12, jitter=0.2, seed=7)
    assert O.hmax(m) > d
    c = I.inv_dist_kernel_c(d)
    off = I.ngon_offsets(32, d) if ball == "ngon" else None
    ref = O.assemble(m, dict(delta=d, ball=ball, outer="dunavant7", inner="dunavant7", kernel="inv_dist", kernel_c=c,
                             ngon_off=off), want_hash=True)
    ctx = nl.nl_create(0)
    try:
        keep = nl._Keep()
        mesh = nl.make_mesh(m, keep)
        cfg = nl.make_config(keep, d, ball, "dunavant7", "dunavant7", "inv_dist", c, off, prec=prec)
        D = nl.nl_assemble(ctx, mesh, cfg)
        G = nl.to_scipy(ctx, D)
        nl.nl_csr_free(ctx, D)
        h, n, q = nl.nl_interactions(ctx, mesh, cfg)
    finally:
        nl.nl_destroy(ctx)
    R = O.to_csr(ref).tocsr()
    R.sort_indices()
    np.testing.assert_array_equal(G.indptr, R.indptr)
    np.testing.assert_array_equal(G.indices, R.indices)
    assert np.abs(G.data - R.data).max() <= TOL[prec] * np.abs(R.data).max()
    np.testing.assert_array_equal(n, ref["count_a"])
    np.testing.assert_array_equal(q, ref["qp_a"])
    np.testing.assert_array_equal(h, ref["hash_a"])
