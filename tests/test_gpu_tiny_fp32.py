"""FP32 path, meshes far smaller than the horizon: every pair is interior, and a row's grid scale is beyond FP32."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ball", ["nocaps", "ngon", "barycenter"])
@pytest.mark.parametrize("size", [1e-3, 1e-7, 1e-9, 1e-12])
def test_mesh_inside_every_ball(ball, size):
    from paper_2005_10775_gb300 import nlfem as nl
    m = I.split_square_mesh(0.0, 1.0, 9, jitter=0.2, seed=3)
    m = dataclasses.replace(m, vx=m.vx * size, vy=m.vy * size)
    d, c = 1.0, I.const_kernel_c(1.0)
    off = I.ngon_offsets(32, d) if ball == "ngon" else None
    ref = O.to_csr(O.assemble(m, dict(delta=d, ball=ball, outer="dunavant7", inner="gauss4", kernel_c=c,
                                      ngon_off=off))).tocsr()
    ref.sort_indices()
    ctx = nl.nl_create(0)
    try:
        keep = nl._Keep()
        D = nl.nl_assemble(ctx, nl.make_mesh(m, keep), nl.make_config(keep, d, ball, "dunavant7", "gauss4", "const", c,
                                                                      off, prec="fp32c"))
        G = nl.to_scipy(ctx, D)
        nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    np.testing.assert_array_equal(G.indptr, ref.indptr)
    np.testing.assert_array_equal(G.indices, ref.indices)
    assert np.abs(G.data - ref.data).max() <= 1e-6 * np.abs(ref.data).max()   # the path's stated accuracy
