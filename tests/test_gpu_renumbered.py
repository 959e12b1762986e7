"""Meshes numbered without locality: a triangle's rows then span the whole mesh, their bitmaps leave the ranked
scatter's 24 KB a warp and the hashed scatter takes them, with the constant kernel's interior pairs formed
from the areas.  One mesh a branch: rows of some 800 columns in FP64 (cached rows by size), as many over
17,000 nodes on the FP32 path (by span), and rows of 1,681 columns (longer than the cached ones)."""
import dataclasses

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


def renumbered(m, seed):
    new = np.random.default_rng(seed).permutation(m.nv)      # new index of each node
    order = np.argsort(new)
    return dataclasses.replace(m, vx=m.vx[order], vy=m.vy[order], tri=np.ascontiguousarray(new[m.tri].astype(np.int32)),
                               node_in_omega=m.node_in_omega[order])


# cells, delta, precision: shared memory of a warp of the ranked scatter (4 sums a column, 24 bytes a word of 32
# nodes) 27, 25, 28 and 55 KB
CASES = [(54, 0.26, "fp64"), (130, 0.108, "fp32c"), (40, 2.0, "fp32c"), (40, 2.0, "fp64")]


def rank_bytes(D, m, prec):
    size = 8 if prec == "fp64" else 4
    row = int(np.diff(D.indptr).max())
    lo, hi = D.indices[D.indptr[:-1]], D.indices[D.indptr[1:] - 1]
    words = int(((hi[m.tri].max(1) - lo[m.tri].min(1)) // 32 + 1).max())
    return 4 * ((row + 3) // 4 * 4) * size + 24 * words, row


@pytest.mark.parametrize("ball", ["nocaps", "barycenter"])
@pytest.mark.parametrize("n,d,prec", CASES)
def test_hashed_scatter(nl, ctx, n, d, prec, ball):
    m = renumbered(I.split_square_mesh(0.0, 1.0, n, jitter=0.2, seed=3), 1)
    c = I.const_kernel_c(d)
    mask = np.zeros(m.nv, np.uint8)
    mask[np.random.default_rng(2).choice(m.nv, 24, replace=False)] = 1    # rows to compare
    ref = O.to_csr(O.assemble(m, dict(delta=d, ball=ball, outer="gauss3", inner="gauss3", kernel_c=c),
                              row_mask=mask)).tocsr()
    keep = nl._Keep()
    mesh = nl.make_mesh(m, keep)
    D = nl.nl_assemble(ctx, mesh, nl.make_config(keep, d, ball, "gauss3", "gauss3", "const", c, prec=prec))
    try:
        for again in range(2):
            G = nl.to_scipy(ctx, D)
            size, row = rank_bytes(G, m, prec)
            assert size > 24 * 1024 and (row > 1022) == (d == 2.0)
            top = np.abs(G.data).max()
            for j in np.nonzero(mask)[0]:
                a, b = G.getrow(j), ref.getrow(j)
                b.sort_indices()
                np.testing.assert_array_equal(a.indices, b.indices)
                assert np.abs(a.data - b.data).max() <= TOL[prec] * top
            nl.nl_assemble_numeric(ctx, D)
    finally:
        nl.nl_csr_free(ctx, D)


@pytest.mark.parametrize("prec", ["fp64", "fp32c"])
def test_batch_of_both_numberings(nl, ctx, prec):
    # one renumbered mesh sends the whole launch to the hashed scatter: both matrices are those of their own
    # assemblies, the well-numbered one's by the ranked scatter
    d = 0.26 if prec == "fp64" else 0.108
    n = 54 if prec == "fp64" else 130
    meshes = [I.split_square_mesh(0.0, 1.0, 24, jitter=0.2, seed=4),
              renumbered(I.split_square_mesh(0.0, 1.0, n, jitter=0.2, seed=3), 1)]
    ds = [0.15, d]
    keep = nl._Keep()
    M = [nl.make_mesh(m, keep) for m in meshes]
    C = [nl.make_config(keep, x, "nocaps", "gauss3", "gauss3", "const", I.const_kernel_c(x), prec=prec) for x in ds]
    alone = []
    for mesh, cfg in zip(M, C):
        D = nl.nl_assemble(ctx, mesh, cfg)
        alone.append(nl.to_scipy(ctx, D))
        nl.nl_csr_free(ctx, D)
    batch, outs = nl.nl_batch_create(ctx, M, C)
    try:
        for again in range(2):
            for D, R, m in zip(outs, alone, meshes):
                G = nl.to_scipy(ctx, D)
                np.testing.assert_array_equal(G.indptr, R.indptr)
                np.testing.assert_array_equal(G.indices, R.indices)
                # FP32: both round the same blocks to the same grids, the interior pairs to the rows' grid here
                assert np.abs(G.data - R.data).max() <= TOL[prec] * np.abs(R.data).max()
            assert rank_bytes(alone[1], meshes[1], prec)[0] > 24 * 1024
            nl.nl_batch_run(ctx, batch)
    finally:
        nl.nl_batch_destroy(ctx, batch)
        for D in outs:
            nl.nl_csr_free(ctx, D)
