"""The local solves and coarse inverses at the edges of their rules.

* Subdomains of a few unknowns, whose matrix rows differ in length (near Neumann edges, in the
  sliced row layout with 32 rows and with one row per slice) and whose solves have one block: F_x and
  the tangent against the oracle under the bounds of test_gpu_parity.py (1e-9; FP32 factors refined to
  1e-10: 1e-7).
* A coarse problem with more dofs than are inverted column by column: the tangent, whose coarse term
  goes through the explicit inverse once a solve has formed it, against the oracle; F_x leaves the
  inverse of A_0(u_0) in place.  FP64 1e-9; FP32 refined to 1e-10 times the condition of A_0 (up to
  1e4 at this size): 1e-6.
* The network's products at sizes that are no multiple of a tile, FP32 within 1e-4 and BF16 within
  2e-2 of the FP64 gradient (the bounds of test_gpu_guess.py).
"""
import numpy as np
import pytest

from oracle import fem, mlp, schwarz as S
from paper_2410_24138_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TIGHT = dict(inner_rtol=1e-13, inner_atol=1e-15)


@pytest.fixture(scope="module")
def nls():
    from paper_2410_24138_gb300 import build, nls as binding
    build.build()
    return binding


def compare(nls, p, coupling, precision, load, scale, tol, opts):
    s = nls.make_solver(p, coupling=coupling, precision=precision, **opts)
    sw = S.Schwarz(p, S.Options(coupling=coupling, **opts))
    rng = np.random.default_rng(4)
    free = fem.free_mask(p)
    u = np.where(free, scale * rng.random(free.size), 0.0)
    Fx, _, st = s.eval_Fx(u, load)
    Fo, sto = sw.evaluate(u, load)
    assert np.all(st == 0)
    assert np.linalg.norm(Fx - Fo) <= 1e-9 * np.linalg.norm(Fo)
    v = np.where(free, rng.random(free.size), 0.0)
    y, yo = s.apply_tangent(v), sw.tangent(sto)(v)
    assert np.linalg.norm(y - yo) <= tol * np.linalg.norm(yo)
    return s


@pytest.mark.parametrize("n,per,overlap", [(3, 1, 1), (4, 2, 1), (7, 3, 1), (9, 2, 2)])
@pytest.mark.parametrize("law", ["p1", "q1"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_small_subdomains(nls, n, per, overlap, law, precision):
    part = I.box_partition(n, per, per)
    if law == "p1":
        p = I.diffusion_problem(n, part, per * per, overlap)
    else:
        p = I.neohooke_problem(n, part, per * per, overlap, traction_max=4.0, load_steps=1)
    compare(nls, p, "one", precision, 0.5, 0.05 if law == "p1" else 0.02 / n, 1e-9 if precision == "fp64" else 1e-7,
            TIGHT)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_inverse_of_many_coarse_dofs(nls, precision):
    p = I.neohooke_problem(96, I.brick_partition(96, 22, 22, 5), 484, 1, traction_max=4.0, load_steps=1)
    s = nls.make_solver(p, coupling="hybrid", precision=precision)
    assert s.sizes().n_coarse_dofs > 2048
    s.close()
    compare(nls, p, "hybrid", precision, 0.3, 0.02 / 96, 1e-9 if precision == "fp64" else 1e-6,
            dict(inner_rtol=1e-12, inner_atol=1e-14))


@pytest.mark.parametrize("B,h1,h2", [(1, 16, 16), (33, 80, 48), (130, 144, 16)])
@pytest.mark.parametrize("bf16,tol", [(False, 1e-4), (True, 2e-2)])
def test_network_products_at_odd_sizes(nls, B, h1, h2, bf16, tol):
    net = nls.GuessNet(h1=h1, h2=h2, seed=3)
    rng = np.random.default_rng(0)
    X = rng.standard_normal((B, net.n_in)).astype(np.float32)
    T = rng.standard_normal((B, net.n_out)).astype(np.float32)
    g, L = net.gradient(X, T, bf16=bf16)
    params = [(W.astype(np.float64), b.astype(np.float64)) for W, b in net.split(net.params())]
    Y, cache = mlp.forward(params, X.astype(np.float64))
    if not bf16:
        Yg = net.forward(X)
        assert np.linalg.norm(Yg - Y) <= 1e-5 * np.linalg.norm(Y)
    for (gW, gb), (rW, rb) in zip(net.split(g), mlp.backward(params, cache, Y, T.astype(np.float64))):
        assert np.linalg.norm(gW - rW) <= tol * np.linalg.norm(rW)
        assert np.linalg.norm(gb - rb) <= tol * max(np.linalg.norm(rb), 1e-30)
