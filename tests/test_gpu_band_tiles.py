"""The tiled band LU (16 x 16 tiles in FP32, 8 x 8 in FP64) at the edges of its tiles and windows.

* Matrix sizes and half bandwidths below, at and just above one, two and several tiles, through
  nls_band_solve with the one-CTA factorization, under the bounds that test_gpu_coarse_factor.py
  derives (entry-by-entry backward error of the factors, forward error on column-dominant
  matrices, the refined solve).
* One subdomain that is so large that the window has no room for the next panel's tiles (11,375
  local unknowns, half bandwidth 66, FP32): F_x and the tangent against the oracle, which solves
  the same local problem with a sparse LU.  F_x = u - w with w the local Newton iterate; both sides
  stop at 1e-12 relative, so they agree to the conditioning of one correction, 1e-9; the tangent of
  a single subdomain is the identity on the free dofs, to the refinement's 1e-10 times the
  condition of the local matrix (about 1e4 on this mesh): 1e-6.
"""
import dataclasses

import numpy as np
import pytest

from oracle import schwarz as S
from paper_2410_24138_gb300 import inputs as I
from test_gpu_coarse_factor import check, column_dominant_band, nls  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,b", [(1, 1), (7, 7), (8, 1), (9, 8), (15, 14), (16, 16), (17, 16), (33, 17), (40, 39),
                                 (65, 32), (130, 49), (257, 105)])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tile_edges(nls, n, b, precision):  # noqa: F811
    prec = nls.PREC_FP32_IR if precision == "fp32" else nls.PREC_FP64
    check(nls, column_dominant_band(n, min(b, max(n - 1, 0)), seed=n + b), prec, nls.COARSE_FACTOR_BAND)


def test_window_without_the_next_panel(nls):  # noqa: F811
    nx, ny = 66, 176
    xy, conn = I.structured_rect_mesh(nx, ny, I.P1_TRI, 1.0, ny / nx)
    i, j = np.arange(xy.shape[0]) % (nx + 1), np.arange(xy.shape[0]) // (nx + 1)
    edge = np.nonzero((i == 0) | (i == nx) | (j == 0) | (j == ny))[0].astype(np.int64)
    p = I.diffusion_problem(2, np.zeros(4, dtype=np.int32), 1, 1)
    p = dataclasses.replace(p, n=nx, xy=xy, conn=conn, dirichlet_nodes=edge,
                            elem_to_sub=np.zeros(conn.shape[0], dtype=np.int32))
    tight = dict(inner_rtol=1e-12, inner_atol=1e-13)
    s = nls.make_solver(p, coupling="one", precision="fp32", **tight)
    assert s.sizes().max_local_dofs == 65 * 175 and s.sizes().max_half_band == 66
    rng = np.random.default_rng(3)
    free = np.ones(xy.shape[0], dtype=bool)
    free[edge] = False
    u = np.where(free, 0.05 * rng.random(xy.shape[0]), 0.0)
    Fx, _, st = s.eval_Fx(u)
    Fo, _ = S.Schwarz(p, S.Options(coupling="one", **tight)).evaluate(u)
    assert np.all(st == 0)
    assert np.linalg.norm(Fx - Fo) <= 1e-9 * np.linalg.norm(Fo)
    v = np.where(free, rng.random(xy.shape[0]), 0.0)
    assert np.linalg.norm(s.apply_tangent(v) - v) <= 1e-6 * np.linalg.norm(v)
