"""The candidate search's cell grid, restated: its indices stay within the grid and its integers within 32 bits for
meshes far smaller than the horizon, of one point, and of parts far from each other."""
import math

import pytest

INT_MAX = 2 ** 31 - 1


def grid(K, delta, rmax, Lx, Ly):
    """nl_prepare_b's grid (mesh.cu)."""
    R = (delta + 2.0 * rmax) * (1.0 + 2e-5)
    L = max(Lx, Ly, 1e-300)
    cs = min(R, L / math.sqrt(max(K / 32.0, 1.0)))
    while (math.floor(Lx / cs) + 1.0) * (math.floor(Ly / cs) + 1.0) > 1073741824.0:
        cs *= 2.0
    nx, ny = math.floor(Lx / cs) + 1, math.floor(Ly / cs) + 1
    return R, cs, nx, ny, int(min(math.ceil(R / cs), float(max(nx, ny))))


@pytest.mark.parametrize("K,delta,rmax,L", [(162, 1.0, 1e-10, 1e-9), (162, 1.0, 1e-13, 1e-12), (1, 1.0, 0.1, 0.0),
                                            (64, 1.0, 0.5, 1e9), (96800, 1.6, 0.1, 32.0), (2, 1.0, 0.1, 0.03)])
def test_reach_fits(K, delta, rmax, L):
    R, cs, nx, ny, m = grid(K, delta, rmax, L, L)
    strip = grid(200000, 1.6, 0.4, 1e5, 1.0)   # a long strip keeps cells of the search radius
    assert strip[1] == strip[0] and strip[2] > 30000 and strip[3] == 1
    assert 1 <= nx * ny <= INT_MAX
    assert nx + m <= INT_MAX                     # cx + g.m in k_candidates
    assert m * cs >= R or m >= max(nx, ny)       # nothing within reach is left out
    for cx in (0, nx // 2, nx - 1):
        assert 0 <= max(cx - m, 0) <= min(cx + m, nx - 1) <= nx - 1
