"""The FP32 near-field rule of the singular kernel (formed by moments) against the FP64 rule (formed point by
point), over its orders: one node, few, the most; a regular and a distorted mesh (many and few panels)."""
import numpy as np
import pytest

from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jitter", [0.0, 0.25])
@pytest.mark.parametrize("duffy_n", [1, 2, 5, 7])
def test_moments_against_points(duffy_n, jitter):
    from paper_2005_10775_gb300 import nlfem as nl
    m = I.split_square_mesh(0.0, 1.0, 9, jitter=jitter, seed=3)
    vals = []
    ctx = nl.nl_create(0)
    try:
        for prec in ("fp64", "fp32c"):
            keep = nl._Keep()
            D = nl.nl_assemble(ctx, nl.make_mesh(m, keep), nl.make_config(
                keep, 0.31, "ngon", "dunavant7", "dunavant7", "inv_dist", 1.0,
                ngon_off=I.ngon_offsets(32, 0.31), prec=prec, duffy_n=duffy_n))
            vals.append(nl.nl_csr_download(ctx, D))
            nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    (rp, ci, v64), (rq, cj, v32) = vals
    assert np.array_equal(rp, rq) and np.array_equal(ci, cj)
    assert np.abs(v32 - v64).max() <= 1e-6 * np.abs(v64).max()   # the FP32 path's stated accuracy
