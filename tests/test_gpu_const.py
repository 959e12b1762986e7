"""The constant kernel's moment path (k_const) at the edges of its walk: polygons of few and many
corners, polygons that are not the regular one, horizons from below a triangle to many, outer points
on vertices and edges, and arc levels on both sides of the FP32 walk's limit, against the FP64 oracle.

Bars: interaction records and pattern bit-exact; values within 1e-12 max|D| (FP64 path: a pair's
block is a few hundred FP64 operations on coordinates of the triangle's own size) and 1e-6 max|D|
(FP32 path, as for every other ball)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32c": 1e-6}


@pytest.fixture(scope="module")
def nl():
    from paper_2005_10775_gb300 import nlfem
    return nlfem


@pytest.fixture(scope="module")
def ctx(nl):
    c = nl.nl_create(0)
    yield c
    nl.nl_destroy(c)


def turned(n, delta, angle):
    """A regular polygon turned by `angle`: its vertices are not R (cos 2 pi k / N, sin 2 pi k / N)."""
    o, c, s = I.ngon_offsets(n, delta), np.cos(angle), np.sin(angle)
    return np.ascontiguousarray(np.stack([c * o[:, 0] - s * o[:, 1], s * o[:, 0] + c * o[:, 1]], 1))


CASES = [
    # ball, cells, delta, jitter, outer, extras
    ("ngon", 14, 0.2, 0.2, "dunavant7", {"off": ("regular", 3)}),
    ("ngon", 14, 0.2, 0.2, "dunavant7", {"off": ("regular", 4)}),
    ("ngon", 14, 0.2, 0.2, "paper7", {"off": ("regular", 7)}),
    ("ngon", 14, 0.2, 0.0, "paper7", {"off": ("regular", 32)}),     # corners on mesh lines
    ("ngon", 14, 0.2, 0.2, "dunavant16", {"off": ("regular", 64)}),
    ("ngon", 10, 0.05, 0.2, "dunavant7", {"off": ("regular", 32)}),  # polygon inside a triangle
    ("ngon", 14, 0.2, 0.2, "dunavant7", {"off": ("turned", 32)}),
    ("ngon", 14, 0.2, 0.2, "switch47", {"off": ("turned", 5)}),
    ("nocaps", 10, 0.05, 0.2, "dunavant7", {}),
    ("approxcaps", 14, 0.2, 0.2, "dunavant7", {"cap_m": 1}),
    ("approxcaps", 10, 0.05, 0.2, "dunavant7", {}),                   # arcs beyond a half circle
    ("approxcaps", 10, 0.05, 0.2, "dunavant7", {"cap_m": 4}),
    ("approxcaps", 14, 0.2, 0.2, "switch47", {"cap_m": 4}),
    ("approxcaps", 14, 0.2, 0.2, "dunavant7", {"cap_m": 8}),         # past the FP32 walk: FP64 regions
    ("exactcaps", 14, 0.2, 0.0, "switch47", {}),
    ("exactcaps", 10, 0.05, 0.2, "dunavant7", {}),
    ("barycenter", 14, 0.2, 0.0, "paper7", {}),
    ("overlap", 14, 0.2, 0.0, "paper7", {}),
]


@pytest.mark.parametrize("ball,n,delta,jitter,outer,kw", CASES)
@pytest.mark.parametrize("prec", ["fp64", "fp32c"])
def test_const_walk_edges(nl, ctx, ball, n, delta, jitter, outer, kw, prec):
    kw = dict(kw)
    off = kw.pop("off", None)
    if off is not None:
        off = I.ngon_offsets(off[1], delta) if off[0] == "regular" else turned(off[1], delta, 0.05)
    m = I.split_square_mesh(-delta, 1.0 + delta, n, jitter=jitter, seed=7 if jitter else None)
    kc = -0.5 * I.const_kernel_c(delta)   # any constant: the paths scale by it, its sign included
    ref = O.assemble(m, dict(delta=delta, ball=ball, outer=outer, inner="gauss4", kernel_c=kc, ngon_off=off,
                             cap_m=kw.get("cap_m", 2)), want_hash=True)
    keep = nl._Keep()
    mesh = nl.make_mesh(m, keep)
    cfg = nl.make_config(keep, delta, ball, outer, "gauss4", "const", kc, off, kw.get("cap_m", 2), prec)
    D = nl.nl_assemble(ctx, mesh, cfg)
    try:
        G = nl.to_scipy(ctx, D)
        stats = (D.n_pairs, D.n_qp_pairs, D.n_inter)
    finally:
        nl.nl_csr_free(ctx, D)
    R = O.to_csr(ref).tocsr()
    R.sort_indices()
    assert stats == (ref["n_pairs"], ref["n_qp_pairs"], ref["n_inter"])
    np.testing.assert_array_equal(G.indptr, R.indptr)
    np.testing.assert_array_equal(G.indices, R.indices)
    assert np.abs(G.data - R.data).max() <= TOL[prec] * np.abs(R.data).max()
    h, c, q = nl.nl_interactions(ctx, mesh, cfg)
    np.testing.assert_array_equal(c, ref["count_a"])
    np.testing.assert_array_equal(q, ref["qp_a"])
    np.testing.assert_array_equal(h, ref["hash_a"])
