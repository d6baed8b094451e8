"""Problems at the edges of what setup accepts.

* A subdomain without unknowns (every node of it and of its overlap pinned): F_x, the tangent and the
  solve against the oracle, under the bounds of test_gpu_parity.py (F_x 1e-9; tangent 1e-9 in FP64 and,
  FP32 factors being refined to 1e-10, 1e-7 in FP32; converged solutions 1e-8 and 1e-6).
* A long thin subdomain beside hundreds of small ones: some 460 coarse dofs meet in it, more than the
  shared memory of an SM holds 2 x 32 rows of, and A_0 is as good as full, which in FP64 also takes the
  coarse inverse's form with one operand buffer (half bandwidth above 430).  F_x and the tangent under the
  same bounds (A_0 has a condition below 100, the global tangent one below 200).
* Device arrays that overlap, in F and in the tangent: the results of separate arrays, bit for bit.
* One subdomain that takes the last of the shared memory that setup accepts (227 KB; the sizes below are
  those of the limit: two FP64 vectors, the larger of the solve vector and a band window, and the rest),
  under the bounds of test_gpu_band_tiles.py for such a subdomain: F_x 1e-9, the tangent, which is the
  identity, 1e-6.
* FP64 and a half bandwidth of 113 (a small mesh numbered so that the first and the last unknown are
  neighbours), where the operand ring would take more threads than the tangent's kernel has: F_x and the
  tangent under the bounds above, and the same bits with the prefetch of the operands off and on.
* A device array longer than the problem: the entries beyond come back as zeros, also in memory that the
  allocator hands out again.
"""
import dataclasses

import numpy as np
import pytest

from oracle import fem, schwarz as S
from paper_2410_24138_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TIGHT = dict(inner_rtol=1e-13, inner_atol=1e-15)


@pytest.fixture(scope="module")
def nls():
    from paper_2410_24138_gb300 import build, nls as binding
    build.build()
    return binding


def random_state(p, scale, seed=4):
    rng = np.random.default_rng(seed)
    free = fem.free_mask(p)
    return np.where(free, scale * rng.random(free.size), 0.0), np.where(free, rng.random(free.size), 0.0)


def compare(s, p, coupling, load, scale, tol, opts=TIGHT):
    sw = S.Schwarz(p, S.Options(coupling=coupling, **opts))
    u, v = random_state(p, scale)
    Fx, _, st = s.eval_Fx(u, load)
    Fo, sto = sw.evaluate(u, load)
    assert np.all(st == 0)
    assert np.linalg.norm(Fx - Fo) <= 1e-9 * np.linalg.norm(Fo)
    y, yo = s.apply_tangent(v), sw.tangent(sto)(v)
    assert np.linalg.norm(y - yo) <= tol * np.linalg.norm(yo)


def pinned_corner():
    """12 x 12 P1 cells in 3 x 3 boxes, overlap 1, every node of [0, 1/2]^2 pinned."""
    p = I.diffusion_problem(12, I.box_partition(12, 3, 3), 9, 1)
    pin = np.nonzero((p.xy <= 0.5).all(axis=1))[0]
    return dataclasses.replace(p, dirichlet_nodes=np.union1d(p.dirichlet_nodes, pin).astype(np.int64))


@pytest.mark.parametrize("coupling", ["one", "add", "hybrid"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_subdomain_without_unknowns(nls, coupling, precision):
    p = pinned_corner()
    s = nls.make_solver(p, coupling=coupling, precision=precision, outer_atol=1e-12, **TIGHT)
    assert s.local_dofs(0)[0].size == 0 and s.local_dofs(8)[0].size > 0
    compare(s, p, coupling, 0.5, 0.05, 1e-9 if precision == "fp64" else 1e-7)
    u, rep = s.solve()
    assert rep.status == 0
    uo, _ = S.plain_newton(p, tol=1e-14)
    assert np.linalg.norm(u - uo) <= (1e-8 if precision == "fp64" else 1e-6) * np.linalg.norm(uo)


def strip_problem(law, boxes):
    """4 x 2 boxes cells: columns 0 and 1 are one subdomain, columns 2 and 3 are boxes of 2 x 2; the left edge is
    clamped."""
    nx, ny = 4, 2 * boxes
    if law == "p1":
        p = I.diffusion_problem(2, np.zeros(4, dtype=np.int32), 1, 1)
    else:
        p = dataclasses.replace(I.neohooke_problem(2, np.zeros(4, dtype=np.int32), 1, 1, traction_max=0.0),
                                traction_edges=None, traction=None)
    xy, conn = I.structured_rect_mesh(nx, ny, p.elem_type, 1.0, ny / nx)
    cell = np.arange(nx * ny)
    sub = np.where(cell % nx < 2, 0, 1 + cell // nx // 2).astype(np.int32)
    return dataclasses.replace(p, n=nx, xy=xy, conn=conn, dirichlet_nodes=np.nonzero(xy[:, 0] == 0)[0].astype(np.int64),
                               elem_to_sub=I.cell_to_elem_partition(sub, p.elem_type), n_sub=1 + boxes, overlap=1)


@pytest.mark.parametrize("law,boxes", [("p1", 460), ("q1", 158)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_subdomain_with_many_coarse_dofs(nls, law, boxes, precision):
    p = strip_problem(law, boxes)
    s = nls.make_solver(p, coupling="hybrid", precision=precision, **TIGHT)
    assert s.sizes().n_coarse_dofs > 454 and s.sizes().coarse_half_band > 430
    compare(s, p, "hybrid", 0.5, 0.02, 1e-9 if precision == "fp64" else 1e-7)


@pytest.mark.parametrize("shift", [0, 1, 37, -1, -500])
def test_overlapping_device_arrays(nls, shift):
    import torch
    p = I.neohooke_problem(24, I.brick_partition(24, 2, 3, 5), 6, 1, traction_max=4.0, load_steps=1)
    s = nls.make_solver(p, coupling="hybrid")
    u, v = random_state(p, 1e-3)
    n, at = u.size, 512
    s.eval_Fx(u, 0.3)
    for call, x, tail in ((s.lib.nls_apply_tangent, v, ()), (s.lib.nls_eval_F, u, (0.3,))):
        want = s.apply_tangent(v) if not tail else s.eval_F(u, 0.3)
        both = torch.zeros(n + 2 * at, dtype=torch.float64, device="cuda")
        both[at:at + n] = torch.from_numpy(x).cuda()
        first = both.data_ptr()
        torch.cuda.synchronize()
        assert call(s.h, first + 8 * at, first + 8 * (at + shift), 1, *tail) == 0
        assert np.array_equal(both[at + shift:at + shift + n].cpu().numpy(), want)


def test_longer_device_arrays(nls):
    import torch
    p = I.diffusion_problem(16, I.box_partition(16, 2, 2), 4, 1)
    s = nls.make_solver(p, coupling="one")
    u, v = random_state(p, 0.05)
    s.eval_Fx(u)
    for call, x in ((s.eval_F, u), (s.apply_tangent, v)):
        long = torch.from_numpy(np.concatenate([x, np.ones(7)])).cuda()
        for _ in range(3):
            used = [torch.full_like(long, 5.0) for _ in range(4)]
            del used
            out = call(long).cpu().numpy()
            assert np.array_equal(out[:x.size], call(x)) and not out[x.size:].any()


def test_subdomain_at_the_limit_of_shared_memory(nls):
    nx, ny = 4, 2635
    p = I.diffusion_problem(2, np.zeros(4, dtype=np.int32), 1, 1)
    xy, conn = I.structured_rect_mesh(nx, ny, I.P1_TRI, 1.0, ny / nx)
    nt, b, limit = xy.shape[0], nx + 1, 227 * 1024
    pinned = np.nonzero(xy[:, 0] == 0)[0].astype(np.int64)
    n = nt - pinned.size

    def up16(k):
        return (k + 15) // 16 * 16

    assert limit - 128 < 8 * (nt + n) + 320 + up16(4 * n) + up16(4 * (b + 10)) + 16 <= limit - 16
    p = dataclasses.replace(p, n=nx, xy=xy, conn=conn, dirichlet_nodes=pinned,
                            elem_to_sub=np.zeros(conn.shape[0], dtype=np.int32), n_sub=1, overlap=1)
    tight = dict(inner_rtol=1e-12, inner_atol=1e-13)
    s = nls.make_solver(p, coupling="one", precision="fp32", **tight)
    assert s.sizes().max_local_dofs == n and s.sizes().max_half_band == b
    u, v = random_state(p, 0.05)
    Fx, _, st = s.eval_Fx(u, 0.05)
    Fo, _ = S.Schwarz(p, S.Options(coupling="one", **tight)).evaluate(u, 0.05)
    assert np.all(st == 0)
    assert np.linalg.norm(Fx - Fo) <= 1e-9 * np.linalg.norm(Fo)
    assert np.linalg.norm(s.apply_tangent(v) - v) <= 1e-6 * np.linalg.norm(v)


def test_widest_band_in_fp64(nls):
    p = I.diffusion_problem(2, np.zeros(4, dtype=np.int32), 1, 1)
    xy, conn = I.structured_rect_mesh(4, 22, I.P1_TRI, 1.0, 5.5)
    n = xy.shape[0] - 1
    old = np.concatenate([[0], np.arange(2, n), [1, n]])  # node 1 becomes the last unknown; the last node is pinned
    new = np.empty(n + 1, dtype=np.int32)
    new[old] = np.arange(n + 1)
    p = dataclasses.replace(p, n=4, xy=xy[old], conn=new[conn], dirichlet_nodes=np.array([n], dtype=np.int64),
                            elem_to_sub=np.zeros(conn.shape[0], dtype=np.int32), n_sub=1, overlap=1)
    got = []
    for dist in (0, 4):
        s = nls.make_solver(p, coupling="one", precision="fp64", l2_prefetch=dist, **TIGHT)
        assert s.sizes().max_half_band == 113 and s.sizes().max_local_dofs == n
        compare(s, p, "one", 0.05, 0.05, 1e-9)
        u, v = random_state(p, 0.05)
        got.append(np.concatenate([s.eval_Fx(u, 0.05)[0], s.apply_tangent(v)]))
    assert np.array_equal(*got)
