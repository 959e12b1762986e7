"""Approxcaps on the FP32 path over the arc levels: the arcs' radius keeps the digits that delta loses in FP32.

Bar: 5e-8 of D in the root mean square.  The roundings of FP32 geometry are independent and leave 2e-8; a radius
of delta rounded to FP32 (4e-8 for delta = 0.15) shifts every region the same way, 9e-8 of D."""
import numpy as np
import pytest

from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap_m", [1, 2, 4, 8, 16])
def test_arc_levels(cap_m):
    from paper_2005_10775_gb300 import nlfem as nl
    m = I.split_square_mesh(0.0, 1.0, 20, jitter=0.2, seed=7)
    d, vals = 0.15, {}
    ctx = nl.nl_create(0)
    try:
        for prec in ("fp64", "fp32c"):
            keep = nl._Keep()
            D = nl.nl_assemble(ctx, nl.make_mesh(m, keep),
                               nl.make_config(keep, d, "approxcaps", "dunavant7", "dunavant7", "const",
                                              I.const_kernel_c(d), None, cap_m, prec=prec))
            vals[prec] = nl.nl_csr_download(ctx, D)[2]
            nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
    e = vals["fp32c"] - vals["fp64"]
    assert np.abs(e).max() <= 1e-6 * np.abs(vals["fp64"]).max()
    assert np.sqrt((e ** 2).mean()) <= 5e-8 * np.sqrt((vals["fp64"] ** 2).mean())
