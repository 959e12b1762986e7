"""What the process's memory pool keeps: 8 GiB as a rule, more while assemblies leave more in use, and 8 GiB again
after smaller ones and after the contexts."""
import ctypes

import pytest

from paper_2005_10775_gb300 import inputs as I

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def threshold():
    cu = ctypes.CDLL("libcuda.so.1")
    pool, v = ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert cu.cuMemPoolGetAttribute(pool, 4, ctypes.byref(v)) == 0   # the release threshold
    return v.value


def test_threshold_follows_use():
    from paper_2005_10775_gb300 import nlfem as nl

    def assemble(ctx, n, d):
        keep = nl._Keep()
        m = I.split_square_mesh(0.0, 1.0, n, jitter=0.2, seed=1)
        return nl.nl_assemble(ctx, nl.make_mesh(m, keep), nl.make_config(keep, d, "nocaps", "dunavant7", "dunavant7",
                                                                         "const", I.const_kernel_c(d), prec="fp64"))

    ctx, other = nl.nl_create(0), nl.nl_create(0)
    try:
        assert threshold() == 8 * GIB
        big = [assemble(ctx, 220, 0.05) for _ in range(2)]   # some 5 GB each
        assert 8 * GIB < threshold() < 64 * GIB
        for D in big:
            nl.nl_csr_free(ctx, D)
        for _ in range(2):
            nl.nl_csr_free(other, assemble(other, 8, 0.2))
        assert threshold() == 8 * GIB
        big = [assemble(ctx, 220, 0.05) for _ in range(2)]
        assert threshold() > 8 * GIB
        for D in big:
            nl.nl_csr_free(ctx, D)
    finally:
        nl.nl_destroy(ctx)
        nl.nl_destroy(other)
    assert threshold() == 8 * GIB
