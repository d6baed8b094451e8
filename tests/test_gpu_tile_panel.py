"""Pivots of the tiled coarse factorization (the panel step of a tile column).

A matrix whose elimination meets an exact zero at one chosen row has to be reported there, whichever
place the row has in the 16- or 8-wide blocks of a diagonal tile.  The matrix is diagonal with a 2 x 2
block [[1, 1], [1, 1]] at rows (r - 1, r): pivot r is 1 - 1 * 1 = 0 without rounding, every other pivot
is 1.  With [[1, 1], [1, 2]] there instead, the factors are whole numbers and come back exactly; the
solution is checked to 10 kappa_inf(A) times the refinement's residual target, kappa_inf = 3 * 3."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nls():
    from paper_2410_24138_gb300 import build, nls as binding
    build.build()
    return binding


def pair_matrix(n, b, r, corner):
    band = np.zeros((n, 2 * b + 1))
    band[:, b] = 1.0
    band[r - 1, b + 1] = band[r, b - 1] = 1.0
    band[r, b] = corner
    return band


@pytest.mark.parametrize("n,b,r", [(300, 130, 1), (300, 130, 7), (300, 130, 8), (300, 130, 15), (300, 130, 16),
                                   (300, 130, 63), (300, 130, 64), (300, 130, 127), (300, 130, 128),
                                   (300, 130, 299), (129, 1, 128), (2, 1, 1)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_pivot_at_each_place_of_a_tile(nls, n, b, r, precision):
    prec = nls.PREC_FP32_IR if precision == "fp32" else nls.PREC_FP64
    with pytest.raises(nls.NLSError) as err:
        nls.band_solve(pair_matrix(n, b, r, 1.0), np.ones(n), precision=prec, method=nls.COARSE_FACTOR_TILES)
    assert err.value.status == -6  # NLS_E_PIVOT
    g = np.arange(1.0, n + 1.0)
    x, F = nls.band_solve(pair_matrix(n, b, r, 2.0), g, precision=prec, method=nls.COARSE_FACTOR_TILES,
                          want_factors=True)
    want = g.copy()
    want[r] = g[r] - g[r - 1]  # L y = g, then U x = y with U = [[1, 1], [0, 1]] at rows (r - 1, r)
    want[r - 1] = g[r - 1] - want[r]
    assert np.array_equal(F, pair_matrix(n, b, r, 1.0))
    assert np.abs(x - want).max() <= 10 * 9 * (1e-10 if precision == "fp32" else 1e-15) * np.abs(want).max()
