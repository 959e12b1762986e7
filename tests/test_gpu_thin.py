"""Thin triangles on the FP32 path: a pair of grid lines so close that rounding a triangle's vertices to FP32
leaves it no area, against the FP64 oracle (the path's stated 1e-6 of max|D|)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def close_lines(n, gap):
    """A uniform n - 1 cell grid on (0, 1)^2 with one more line `gap` cells above its middle one."""
    m = I.split_square_mesh(0.0, 1.0, n)
    k = n // 2
    y = np.arange(n) / (n - 1.0)
    y = np.concatenate([y[:k + 1], [y[k] + gap / (n - 1.0)], y[k + 1:]])
    return I.Mesh(vx=m.vx, vy=y[np.rint(m.vy * n).astype(int)], tri=m.tri, node_in_omega=m.node_in_omega,
                  elem_in_omega=m.elem_in_omega, h=m.h, lo=0.0, hi=1.0, n=n)


@pytest.mark.parametrize("delta", [0.17, 0.05])   # above and below the triangles' diameter
@pytest.mark.parametrize("ball", ["nocaps", "exactcaps", "ngon"])
@pytest.mark.parametrize("gap", [1e-4, 1e-6, 1e-8, 1e-10])
def test_thin_triangles(ball, gap, delta):
    from paper_2005_10775_gb300 import nlfem as nl
    m = close_lines(16, gap)
    c = I.const_kernel_c(delta)
    off = I.ngon_offsets(32, delta) if ball == "ngon" else None
    ref = O.to_csr(O.assemble(m, dict(delta=delta, ball=ball, outer="dunavant7", inner="dunavant7", kernel_c=c,
                                      ngon_off=off))).tocsr()
    ref.sort_indices()
    ctx = nl.nl_create(0)
    try:
        keep = nl._Keep()
        D = nl.nl_assemble(ctx, nl.make_mesh(m, keep), nl.make_config(keep, delta, ball, "dunavant7", "dunavant7",
                                                                      "const", c, off, prec="fp32c"))
        G = nl.to_scipy(ctx, D)
        nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    np.testing.assert_array_equal(G.indptr, ref.indptr)
    np.testing.assert_array_equal(G.indices, ref.indices)
    assert np.abs(G.data - ref.data).max() <= 1e-6 * np.abs(ref.data).max()
