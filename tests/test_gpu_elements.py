"""The Neo-Hooke element routines far from the identity: F(u) with J = det F between 1e-3 and 1e3.

The library takes log J and 1 / J from a table step (two binades around 1 need no exponent, the
others do), the oracle from the math library.  Both sum the same Gauss-point terms in FP64: the
terms of one node's residual are at most S = max_q w (mu |F| + |c| |F^-1|) |grad N| each, every one
carries a few roundings (F, J, 1 / J and log J: below 2e-15 relative to S), 16 of them meet in a node
and cancel, so the two sides differ by at most 16 x 2e-15 S < 1e-13 S, S bounded by the largest
node sum of the absolute terms."""
import numpy as np
import pytest

from oracle import fem
from paper_2410_24138_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch", [0.032, 0.3, 0.86, 0.87, 1.0, 1.22, 1.23, 3.0, 31.0])
def test_residual_at_large_stretch(stretch):
    from paper_2410_24138_gb300 import build, nls
    build.build()
    p = I.neohooke_problem(12, I.brick_partition(12, 2, 2, 5), 4, 1, traction_max=4.0)
    s = nls.make_solver(p, coupling="one")
    rng = np.random.default_rng(int(100 * stretch))
    u = ((stretch - 1.0) * p.xy + 0.02 * stretch / 12 * rng.standard_normal(p.xy.shape)).reshape(-1)
    F = s.eval_F(u, 0.3)
    Fo = fem.global_residual(fem.Model(p), u, 0.3)
    mu, lam = 210.0 / 2.6, 210.0 * 0.3 / (1.3 * 0.4)
    c = abs(mu - lam * np.log(stretch ** 2))
    S = 4 * (1.0 / 12) * (mu * stretch + c / stretch)  # four elements meet; w |grad N| ~ h
    assert np.max(np.abs(F - Fo)) <= 1e-13 * max(S, np.max(np.abs(Fo)))
