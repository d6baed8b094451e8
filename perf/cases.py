"""Performance cases of the nonlinear Schwarz solver, through its public entry points.

Two families of problems, both on n x n cells of the unit square cut into per x per uneven bricks
with an overlap of two element layers:

* ``p1``: nonlinear diffusion (Eq. 1) on triangles, log-normal coefficient field k (or k = 1),
  one constant source per instance in [0.5, 2];
* ``q1``: Neo-Hooke elasticity (Eq. 2) on quadrilaterals, left edge clamped, vertical dead load on
  the right edge, ramped over ``load_steps``.

Kinds of a case, in the order in which a solve uses them:

* ``residual``     F(u) of Eq. 3, on device tensors: what a line search or a monitor calls;
* ``corrections``  F_x(u) of Eqs. 5 and 11: the batched subdomain Newton solves, and with the
                   two-level coupling the coarse Newton solve, leaving the tangent's factors;
* ``tangent``      y = DF_x(u) v of Eqs. 6 and 12: one per GMRES iteration;
* ``solve``        the whole method from u = 0;
* ``infer``, ``train``  the learned initial guess: the network on a batch of subdomains, and Adam
                   steps (forward, backward, update) on harvested pairs.

``exact`` is plain 64-bit torch on the structured grid: every problem is a batch of rectangular
windows of nodes, every linear system is solved by block elimination along the window's lines.
"""
import math

import numpy as np
import torch

from paper_2410_24138_gb300 import inputs, nls

TRACTION = 8.0  # dead load of the Neo-Hooke workloads at load factor 1


def listed():
    return [
        # one residual of the 64 x 64 plain problem: the smallest call there is, all latency
        dict(name="residual-p1-64", kind="residual", law="p1", n=64, per=4, rough=False),
        # one residual of an elastic problem of a few hundred thousand dofs
        dict(name="residual-q1-384", kind="residual", law="q1", n=384, per=12),
        # the subdomain solves of the log-normal diffusion workload, two-level, FP32 factors + refinement
        dict(name="corrections-p1-512", kind="corrections", law="p1", n=512, per=16, coupling="hybrid",
             precision="fp32", rough=True),
        # the same step of the elastic workload in the plain FP64 form, one-level, an odd mesh
        dict(name="corrections-q1-255-fp64", kind="corrections", law="q1", n=255, per=9, coupling="one",
             precision="fp64"),
        # one GMRES iteration's operator on the log-normal diffusion workload
        dict(name="tangent-p1-512", kind="tangent", law="p1", n=512, per=16, coupling="hybrid", precision="fp32",
             rough=True),
        # and on the elastic workload: subdomains of 32 x 32 cells, as in the 512 and 2048 meshes
        dict(name="tangent-q1-384", kind="tangent", law="q1", n=384, per=12, coupling="hybrid", precision="fp32"),
        # the plain method on its smallest workload: many short launches, few subdomains
        dict(name="solve-p1-64-fp64", kind="solve", law="p1", n=64, per=4, coupling="hybrid", precision="fp64",
             rough=False, load_steps=1),
        # the chosen form on a diffusion mesh of a quarter million dofs
        dict(name="solve-p1-512", kind="solve", law="p1", n=512, per=16, coupling="hybrid", precision="fp32",
             rough=True, load_steps=1),
        # the chosen form on the elastic workload, subdomains of 32 x 32 cells, five load steps
        dict(name="solve-q1-384", kind="solve", law="q1", n=384, per=12, coupling="hybrid", precision="fp32",
             load_steps=5),
        # many small subdomains: a coarse problem wide enough for the tiled factorization
        dict(name="solve-q1-256-many", kind="solve", law="q1", n=256, per=32, coupling="hybrid", precision="fp32",
             load_steps=2),
        # the proposals of one outer iteration: the network on every subdomain's inputs
        dict(name="infer-1024", kind="infer", net="scalar", batch=1024, hidden=512),
        # a stretch of the network's training: BF16 operands, batches of 256 pairs
        dict(name="train-256", kind="train", net="scalar", batch=256, hidden=512, steps=40),
    ]


def draw(rng):
    kind = rng.choice(["residual", "corrections", "tangent", "solve", "solve", "infer", "train"])
    if kind in ("infer", "train"):
        hidden = 16 * rng.randint(4, 32)
        if kind == "infer":
            return dict(kind=kind, net=rng.choice(["scalar", "displacement"]),
                        batch=int(round(16 * 64 ** rng.random())) + rng.randint(0, 3), hidden=hidden)
        return dict(kind=kind, net="scalar", batch=rng.randint(32, 256), hidden=hidden, steps=rng.randint(10, 40))
    law = rng.choice(["p1", "q1"])
    top = {"p1": 512, "q1": 384}[law]
    n = int(round(48 * (top / 48.0) ** rng.random()))
    per = max(2, int(round(n / (8.0 * 4.0 ** rng.random()))))  # subdomains of 8 to 32 cells a side
    if law == "q1":
        per = min(per, 36)
    case = dict(kind=kind, law=law, n=n, per=per)
    if law == "p1":
        case["rough"] = rng.random() < 0.7
    if kind != "residual":
        case["precision"] = rng.choice(["fp32", "fp32", "fp64"])
        case["coupling"] = rng.choice(["one", "add", "hybrid", "hybrid"] if kind != "solve" else ["add", "hybrid"])
    if kind == "solve":
        case["load_steps"] = 1 if law == "p1" else rng.randint(1, 4)
    return case


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------

def _fields(case, seed):
    """Cell coefficients k and f of a diffusion case."""
    n = case["n"]
    gen = inputs.splitmix64(seed ^ 0x5DEECE66D)
    f = 0.5 + 1.5 * float(inputs.uniform01(gen, 1)[0])
    k = np.exp(inputs.gaussian_random_field(n, seed, ell=1.0 / 16.0)) if case["rough"] else np.ones(n * n)
    return k, np.full(n * n, f)


def _traction(seed):
    """Dead load of an elastic case: the workload's, or somewhat less."""
    return TRACTION * (0.75 + 0.25 * float(inputs.uniform01(inputs.splitmix64(seed), 1)[0]))


def _partition(case):
    return inputs.brick_partition(case["n"], case["per"], case["per"], inputs.PARTITION_SEED)


def _problem(case, seed):
    n, per = case["n"], case["per"]
    if case["law"] == "p1":
        k, f = _fields(case, seed)
        return inputs.diffusion_problem(n, _partition(case), per * per, 2, k_cell=k, f_cell=f)
    return inputs.neohooke_problem(n, _partition(case), per * per, 2, _traction(seed), case.get("load_steps", 1))


def _state(case, seed):
    """A point the outer iteration meets: a smooth state of the solution's size that satisfies the
    Dirichlet data, with a smaller short-wave part (node-wise rough only as far as h allows)."""
    n, d = case["n"], _ndof(case)
    rng = np.random.RandomState(seed % (1 << 31))
    x = np.arange(n + 1) / n
    X, Y = np.meshgrid(x, x)
    if d == 1:
        u = (0.05 + 0.05 * rng.rand()) * np.sin(np.pi * X) * np.sin(np.pi * Y)
        u += 0.01 * np.sin((2 + rng.randint(3)) * np.pi * X) * np.sin((3 + rng.randint(3)) * np.pi * Y)
        u += (0.02 / n) * rng.standard_normal(u.shape)
        u[0] = u[-1] = u[:, 0] = u[:, -1] = 0.0
        return u.reshape(-1)
    tip = 0.05 + 0.03 * rng.rand()  # a bending beam and small waves
    ux = tip * (Y - 0.5) * X * (2.0 - X) + 0.004 * np.sin((1 + rng.randint(3)) * np.pi * X) * np.cos(np.pi * Y)
    uy = -tip * X * X * (3.0 - X) / 2.0 + 0.004 * np.sin(np.pi * X) * np.sin((1 + rng.randint(3)) * np.pi * Y)
    u = np.stack([ux, uy], -1) + (0.002 / n) * rng.standard_normal((n + 1, n + 1, 2))
    u[:, 0] = 0.0
    return u.reshape(-1)


def _direction(case, seed):
    """A Krylov vector: smooth and rough parts of comparable size, zero on the Dirichlet dofs."""
    n, d = case["n"], _ndof(case)
    rng = np.random.RandomState((seed + 77) % (1 << 31))
    x = np.arange(n + 1) / n
    X, Y = np.meshgrid(x, x)
    v = np.stack([np.sin(np.pi * (1 + rng.randint(4)) * X + rng.rand()) * np.sin(np.pi * (1 + rng.randint(4)) * Y)
                  for _ in range(d)], -1) + 0.3 * rng.standard_normal((n + 1, n + 1, d))
    v[:, 0] = 0.0
    if d == 1:
        v[0] = v[-1] = v[:, -1] = 0.0
    return (v / np.linalg.norm(v)).reshape(-1)


def _ndof(case):
    return 1 if case["law"] == "p1" else 2


def _load(case):
    return 1.0 if case["law"] == "p1" else 0.2  # an elastic state of the first load step


def _net(case, capacity=0):
    kind = nls.GUESS_KIND_DISPLACEMENT if case["net"] == "displacement" else nls.GUESS_KIND_SCALAR
    return nls.GuessNet(h1=case["hidden"], h2=case["hidden"], seed=11, capacity=capacity, kind=kind)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "infer":
        net = _net(case)
        X = np.random.RandomState(seed % (1 << 31)).standard_normal((case["batch"], net.n_in)).astype(np.float32)
        return dict(case=case, net=net, X=X)
    if kind == "train":
        small = dict(law="p1", n=96, per=12, rough=True)
        net = _net(case, capacity=2000)
        s = nls.make_solver(_problem(small, seed), coupling="hybrid")
        nls.attach_guess(s, net, nls.GUESS_HARVEST)
        for more in range(2):  # pairs of two coefficient fields
            if more:
                k, f = _fields(small, seed + 1000)
                s.set_coefficients(np.repeat(k, 2), np.repeat(f, 2))
            s.solve()
        s.close()
        return dict(case=case, net=net)
    prob = _problem(case, seed)
    one = case.get("coupling", "one")
    s = nls.make_solver(prob, coupling=one, precision=case.get("precision", "fp32"))
    state = dict(case=case, solver=s)
    if kind == "solve":
        state["u"] = torch.zeros(prob.n_nodes * prob.ndof, dtype=torch.float64, device="cuda")
        return state
    state["u"] = torch.from_numpy(_state(case, seed)).cuda()
    if kind == "tangent":
        s.eval_Fx(state["u"], _load(case))
        state["v"] = torch.from_numpy(_direction(case, seed)).cuda()
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "residual":
        return state["solver"].eval_F(state["u"], _load(case))
    if kind == "corrections":
        Fx, its, status = state["solver"].eval_Fx(state["u"], _load(case))
        return dict(Fx=Fx, its=its, status=status)
    if kind == "tangent":
        return state["solver"].apply_tangent(state["v"])
    if kind == "solve":
        u, _ = state["solver"].solve(state["u"].zero_())
        return u
    if kind == "infer":
        return state["net"].forward(state["X"])
    losses = state["net"].train(case["steps"], batch=case["batch"], lr=1e-3, seed=7)
    return dict(losses=losses, params=state["net"].params())


def work(case):
    """Bytes and operations of one pass that no form of the method can do without (estimates where an
    iteration count enters: two outer iterations per load step of ten operator applications each)."""
    kind = case["kind"]
    if kind in ("infer", "train"):
        ni, no = (nls.GUESS_FEATURES, nls.GUESS_OUTPUTS) if case["net"] == "scalar" else (
            nls.GUESS_FEATURES_DISP, nls.GUESS_OUTPUTS_DISP)
        h, B = case["hidden"], case["batch"]
        weights = ni * h + h * h + h * no
        if kind == "infer":
            return dict(bytes=4.0 * (weights + B * (ni + no)), flops=2.0 * B * weights)
        return dict(bytes=case["steps"] * 4.0 * (7 * weights + B * (ni + no)), flops=case["steps"] * 6.0 * B * weights)
    n, per, d = case["n"], case["per"], _ndof(case)
    N = (n + 1) ** 2 * d
    mesh = (n + 1) ** 2 * 16 + n * n * (2 * 12 + 2 * 8 if d == 1 else 16)  # coordinates, connectivity, coefficients
    element = n * n * (2 * 40 if d == 1 else 400)  # operations of all element residuals
    residual = dict(bytes=2 * 8 * N + mesh, flops=element)
    if kind == "residual":
        return residual
    fb = 4 if case["precision"] == "fp32" else 8
    side = n / per + 3  # nodes of a subdomain with its overlap, per side
    nl, b = side * side * d, side * d + d - 1
    rows = per * per * nl
    nnz = rows * (7 if d == 1 else 18)
    factor, lu = rows * (2 * b + 1), rows * 2 * b * b
    jac = (n * n * (2 * 80 if d == 1 else 1000)) * (side * per / n) ** 2
    operator = dict(bytes=factor * fb + nnz * 12 + 3 * 8 * N, flops=2.0 * (factor + nnz))
    if kind == "tangent":
        return operator
    fx = dict(bytes=residual["bytes"] + factor * fb + nnz * 8, flops=lu + jac + 2 * element)
    if kind == "corrections":
        return fx
    outer = 2 * case["load_steps"]
    return {q: outer * (fx[q] + 10 * operator[q]) for q in ("bytes", "flops")}


# ----------------------------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ----------------------------------------------------------------------------------------------
CORNERS = ((0, 0), (0, 1), (1, 1), (1, 0))  # (dy, dx) of a cell's nodes, counter-clockwise
MU, LAM = 210.0 / 2.6, 210.0 * 0.3 / (1.3 * 0.4)


def _cells(law, h, U, k, tri, tangent):
    """Cell residuals [..., 4, d] and tangents [..., 4 d, 4 d] of nodal values U [..., H, W, d] on
    square cells of side h.  ``tri`` [..., H-1, W-1, 2] says which triangles (p1) or cells (q1) count."""
    u = torch.stack([U[..., dy:U.shape[-3] - 1 + dy, dx:U.shape[-2] - 1 + dx, :] for dy, dx in CORNERS], -2)
    r = torch.zeros_like(u)
    K = u.new_zeros(u.shape[:-2] + (4 * u.shape[-1],) * 2) if tangent else None
    if law == "p1":
        for which, (nodes, grads) in enumerate((((0, 1, 2), ((-1, 0), (1, -1), (0, 1))),
                                                ((0, 2, 3), ((0, -1), (1, 0), (-1, 1))))):
            on = tri[..., which] * k
            w = [u[..., a, 0] for a in nodes]
            g = torch.tensor(grads, dtype=U.dtype, device=U.device) / h
            grad = [sum(w[a] * g[a, i] for a in range(3)) for i in range(2)]
            mid = [(w[0] + w[1]) / 2, (w[1] + w[2]) / 2, (w[2] + w[0]) / 2]
            area3 = h * h / 6
            Q = area3 * (3 + sum(m * m for m in mid))
            dQ = [area3 * (mid[0] + mid[2]), area3 * (mid[0] + mid[1]), area3 * (mid[1] + mid[2])]
            for a in range(3):
                flux = grad[0] * g[a, 0] + grad[1] * g[a, 1]
                r[..., nodes[a], 0] += on * Q * flux
                if tangent:
                    for b in range(3):
                        K[..., nodes[a], nodes[b]] += on * (Q * (g[a] @ g[b]) + flux * dQ[b])
        return r, K
    q = 1 / math.sqrt(3)
    for s, t in ((-q, -q), (q, -q), (q, q), (-q, q)):
        g = torch.tensor([[-(1 - t), -(1 - s)], [1 - t, -(1 + s)], [1 + t, 1 + s], [-(1 + t), 1 - s]],
                         dtype=U.dtype, device=U.device) / (2 * h)
        F = torch.einsum("...ai,aj->...ij", u, g) + torch.eye(2, dtype=U.dtype, device=U.device)
        det = F[..., 0, 0] * F[..., 1, 1] - F[..., 0, 1] * F[..., 1, 0]
        det = torch.where(tri[..., 0] > 0, det, torch.ones_like(det))  # cells that do not count may be folded
        inv = torch.stack([torch.stack([F[..., 1, 1], -F[..., 0, 1]], -1),
                           torch.stack([-F[..., 1, 0], F[..., 0, 0]], -1)], -2) / det[..., None, None]
        c = MU - LAM * torch.log(det)
        p = torch.einsum("aj,...ji->...ai", g, inv)
        w = tri[..., 0] * (h * h / 4)
        r += w[..., None, None] * (MU * torch.einsum("...ij,aj->...ai", F, g) - c[..., None, None] * p)
        if tangent:
            T = (LAM * torch.einsum("...ai,...bk->...aibk", p, p)
                 + c[..., None, None, None, None] * torch.einsum("...ak,...bi->...aibk", p, p))
            T = T + MU * torch.einsum("ab,ik->aibk", g @ g.T, torch.eye(2, dtype=U.dtype, device=U.device))
            K += w[..., None, None] * T.reshape(K.shape)
    return r, K


def _to_nodes(r):
    """Sum of cell contributions [..., Hc, Wc, 4, d] at the nodes."""
    Hc, Wc = r.shape[-4], r.shape[-3]
    out = r.new_zeros(r.shape[:-4] + (Hc + 1, Wc + 1, r.shape[-1]))
    for a, (dy, dx) in enumerate(CORNERS):
        out[..., dy:Hc + dy, dx:Wc + dx, :] += r[..., a, :]
    return out


def _times(K, V):
    """The operator with cell tangents K [B, Hc, Wc, 4 d, 4 d] on V [B, H, W, d, m] (zero extension)."""
    H, W, d, m = V.shape[1:]
    v = torch.stack([V[:, dy:H - 1 + dy, dx:W - 1 + dx] for dy, dx in CORNERS], 3)
    y = (K @ v.reshape(v.shape[:3] + (4 * d, m))).reshape(v.shape[:3] + (4, d * m))
    return _to_nodes(y).reshape(V.shape)


def _block_solve(K, mask, rhs):
    """x with J x = rhs on the nodes of mask [B, H, W] (x = 0 elsewhere), J from cell tangents; rhs and
    x [B, H, W, d, m].  Block elimination without exchange across the lines of the window."""
    B, H, W, d, m = rhs.shape
    T = [K.new_zeros(B, H, W, d, W, d) for _ in range(3)]  # couplings to the line before, own, after
    Kc = K.reshape(B, H - 1, W - 1, 4, d, 4, d)
    for a, (ya, xa) in enumerate(CORNERS):
        for b, (yb, xb) in enumerate(CORNERS):
            off = xb - xa
            diag = T[yb - ya + 1].diagonal(off, 2, 4)  # [B, H, d, d, positions]
            first = xa if off >= 0 else xa - 1  # position of the first cell's pair on that diagonal
            diag[:, ya:H - 1 + ya, :, :, first:first + W - 1] += Kc[:, :, :, a, :, b, :].permute(0, 1, 3, 4, 2)
    on = mask[..., None].expand(B, H, W, d).reshape(B, H, W * d)
    T = [t.reshape(B, H, W * d, W * d) for t in T]
    keep = on[:, :, :, None] & on[:, :, None, :]
    T[1] = T[1] * keep + torch.diag_embed((~on).to(K.dtype))
    rhs = torch.where(on[..., None], rhs.reshape(B, H, W * d, m), torch.zeros((), dtype=K.dtype, device=K.device))
    up, y = [None] * H, [None] * H
    for i in range(H):
        D, g = T[1][:, i], rhs[:, i]
        if i:
            low = T[0][:, i] * (on[:, i, :, None] & on[:, i - 1, None, :])
            D, g = D - low @ up[i - 1], g - low @ y[i - 1]
        if i + 1 < H:
            right = T[2][:, i] * (on[:, i, :, None] & on[:, i + 1, None, :])
            z = torch.linalg.solve(D, torch.cat([right, g], -1))
            up[i], y[i] = z[..., :W * d], z[..., W * d:]
        else:
            y[i] = torch.linalg.solve(D, g)
    for i in range(H - 2, -1, -1):
        y[i] = y[i] - up[i] @ y[i + 1]
    return torch.stack(y, 1).reshape(B, H, W, d, m)


class _Grid:
    """The discrete problem of a case on its structured grid."""

    def __init__(self, case, seed):
        self.case, self.law, self.n, self.d = case, case["law"], case["n"], _ndof(case)
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        n, h = self.n, 1.0 / case["n"]
        self.h = h
        self.sub = torch.from_numpy(_partition(case).reshape(n, n)).long().to(self.dev)
        self.k = torch.ones(n, n, dtype=torch.float64, device=self.dev)
        self.load = torch.zeros(n + 1, n + 1, self.d, dtype=torch.float64, device=self.dev)
        self.free = torch.ones(n + 1, n + 1, dtype=torch.bool, device=self.dev)
        self.free[:, 0] = False
        if self.law == "p1":
            k, f = _fields(case, seed)
            self.k = torch.from_numpy(k.reshape(n, n)).to(self.dev)
            share = float(f[0]) * h * h / 6
            for a, triangles in enumerate((2, 1, 2, 1)):
                dy, dx = CORNERS[a]
                self.load[dy:n + dy, dx:n + dx, 0] += triangles * share
            self.free[:, -1] = self.free[0] = self.free[-1] = False
        else:
            self.load[:, -1, 1] -= _traction(seed) * h
            self.load[0, -1, 1] /= 2
            self.load[-1, -1, 1] /= 2
        self.whole = (torch.zeros(1, dtype=torch.long, device=self.dev),) * 2 + (n + 1, n + 1)
        self.all_cells = torch.ones(1, n, n, 2, dtype=torch.float64, device=self.dev)

    # -- windows: (first row [B], first column [B], rows, columns), nodes outside the mesh allowed
    def at(self, win, field, outside=0):
        j0, i0, H, W = win
        J = j0[:, None, None] + torch.arange(H, device=self.dev)[None, :, None]
        I = i0[:, None, None] + torch.arange(W, device=self.dev)[None, None, :]
        ok = (J >= 0) & (I >= 0) & (J < field.shape[0]) & (I < field.shape[1])
        got = field[J.clamp(0, field.shape[0] - 1), I.clamp(0, field.shape[1] - 1)]
        return torch.where(ok.reshape(ok.shape + (1,) * (got.dim() - 3)), got, torch.full_like(got, outside))

    def cells(self, win, U, tri, tangent):
        k = self.at((win[0], win[1], win[2] - 1, win[3] - 1), self.k)
        return _cells(self.law, self.h, U, k, tri, tangent)

    def residual(self, U, load):
        """F(u) on the grid, zero on the Dirichlet nodes."""
        r, _ = self.cells(self.whole, U[None], self.all_cells, False)
        return torch.where(self.free[..., None], _to_nodes(r)[0] - load * self.load, torch.zeros_like(U))

    def tangent(self, U):
        return self.cells(self.whole, U[None], self.all_cells, True)[1]

    # -- overlapping subdomains
    def subdomains(self, layers=2):
        """Windows that hold every overlapping subdomain and a ring of nodes; which triangles are in it;
        which nodes carry its unknowns; which of them it owns."""
        n, count = self.n, self.case["per"] ** 2
        where = [torch.nonzero(self.sub == s) for s in range(count)]
        lo = torch.stack([w.min(0).values for w in where])
        hi = torch.stack([w.max(0).values for w in where])
        H, W = ((hi - lo).max(0).values + 2 + 2 * layers + 2).tolist()
        win = (lo[:, 0] - layers - 1, lo[:, 1] - layers - 1, H, W)
        cell = (win[0], win[1], H - 1, W - 1)
        exists = self.at(cell, torch.ones_like(self.sub), 0) > 0
        own = self.at(cell, self.sub, -1) == torch.arange(count, device=self.dev)[:, None, None]
        tri = torch.stack([own, own], -1)
        halves = ((0, 1, 2), (0, 2, 3)) if self.law == "p1" else ((0, 1, 2, 3),) * 2

        def touched(t):
            out = torch.zeros(count, H, W, dtype=torch.bool, device=self.dev)
            for w in range(2):
                for a in halves[w]:
                    dy, dx = CORNERS[a]
                    out[:, dy:H - 1 + dy, dx:W - 1 + dx] |= t[..., w]
            return out

        def reached(nodes):
            return torch.stack([torch.stack([nodes[:, dy:H - 1 + dy, dx:W - 1 + dx] for dy, dx in
                                             (CORNERS[a] for a in halves[w])]).any(0) & exists for w in range(2)], -1)

        for _ in range(layers):
            tri = reached(touched(tri))
        unknown = touched(tri) & ~touched(exists[..., None] & ~tri) & self.at(win, self.free, False)
        first = torch.full((n + 1, n + 1), 1 << 30, dtype=torch.long, device=self.dev)
        for dy, dx in CORNERS:
            first[dy:n + dy, dx:n + dx] = torch.minimum(first[dy:n + dy, dx:n + dx], self.sub)
        owned = unknown & (self.at(win, first, -1) == torch.arange(count, device=self.dev)[:, None, None])
        return win, tri.double(), unknown, owned

    def local_newton(self, win, tri, unknown, U, load, rtol=1e-5, atol=1e-11):
        """The converged local states (whole windows) of Eq. 4 at U, with the stopping rule of the solves."""
        w, f, on = self.at(win, U), load * self.at(win, self.load), unknown[..., None]

        def norm(x):
            r = (_to_nodes(self.cells(win, x, tri, False)[0]) - f) * on
            size = r.flatten(1).norm(dim=1)
            return r, torch.where(size.isfinite(), size, torch.full_like(size, math.inf))

        r, rn = norm(w)
        tol = torch.clamp(rtol * rn, min=atol)
        for _ in range(50):
            todo = rn > tol
            if not todo.any():
                return w
            K = self.cells(win, w, tri, True)[1]
            s = _in_parts(K, unknown, r[..., None])[..., 0]
            alpha = torch.ones_like(rn)
            for _ in range(10):
                t = w - (alpha * todo)[:, None, None, None] * s
                rt, rtn = norm(t)
                bad = todo & ~(rtn <= (1 - 1e-4 * alpha) * rn)
                if not bad.any():
                    break
                alpha = torch.where(bad, alpha / 2, alpha)
            w, r, rn = t, rt, rtn
        return w

    def paste(self, win, owned, part):
        out = torch.zeros(self.n + 1, self.n + 1, self.d, dtype=torch.float64, device=self.dev)
        b, j, i = torch.nonzero(owned, as_tuple=True)
        out[win[0][b] + j, win[1][b] + i] = part[b, j, i]
        return out

    # -- the coarse space
    def basis(self):
        """P_0 as [nodes y, nodes x, d, N0]."""
        n, d, law = self.n, self.d, self.law
        sub, free = self.sub.cpu().numpy(), self.free.cpu().numpy()
        cells = np.full((n + 2, n + 2), -1)
        cells[1:-1, 1:-1] = sub
        four = np.stack([cells[dy:n + 1 + dy, dx:n + 1 + dx] for dy in (0, 1) for dx in (0, 1)], -1)
        mixed = np.zeros((n + 1, n + 1), bool)
        for a in range(4):
            for b in range(a):
                mixed |= (four[..., a] != four[..., b]) & (four[..., a] >= 0) & (four[..., b] >= 0)
        sets = {(int(j), int(i)): frozenset(int(s) for s in four[j, i] if s >= 0) for j, i in np.argwhere(mixed)}
        near = [(0, 1), (1, 0), (0, -1), (-1, 0)] + ([(1, 1), (-1, -1)] if law == "p1" else [])
        comps, seen = [], set()
        for v in sets:  # row by row, so components come by their smallest node
            if v in seen:
                continue
            seen.add(v)
            part, todo = [], [v]
            while todo:
                p = todo.pop()
                part.append(p)
                for dj, di in near:
                    q = (p[0] + dj, p[1] + di)
                    if q in sets and q not in seen and sets[q] == sets[v] and free[q] == free[v]:
                        seen.add(q)
                        todo.append(q)
            comps.append((np.array(part, float), sets[v], bool(free[v]), part))
        by_sub = {}
        for c in comps:
            by_sub.setdefault(min(c[1]), [])
            for s in c[1]:
                by_sub.setdefault(s, []).append(c)
        top = [c for c in comps if c[2] and not any(o[2] and o[1] > c[1] for o in by_sub[min(c[1])])]
        index = {id(c): q for q, c in enumerate(top)}
        own = {p: q for q, c in enumerate(top) for p in c[3]}
        modes = 1 if d == 1 else 3
        P = np.zeros((n + 1, n + 1, d, modes * len(top)))
        for v, s in sets.items():
            if not free[v]:
                continue
            if v in own:
                phi = {own[v]: 1.0}
            else:
                above = [c for c in by_sub[min(s)] if s <= c[1] and (not c[2] or id(c) in index)]
                inverse = [1.0 / (np.hypot(c[0][:, 0] - v[0], c[0][:, 1] - v[1]).min() * self.h) for c in above]
                phi = {index[id(c)]: w / sum(inverse) for c, w in zip(above, inverse) if c[2]}
            for q, value in phi.items():
                if d == 1:
                    P[v + (0, q)] = value
                else:
                    cy, cx = top[q][0].mean(0)
                    P[v + (0, 3 * q)] = P[v + (1, 3 * q + 1)] = value
                    P[v + (0, 3 * q + 2)] = -value * (v[0] - cy) * self.h
                    P[v + (1, 3 * q + 2)] = value * (v[1] - cx) * self.h
        P = torch.from_numpy(P).to(self.dev)
        # energy-minimising extension into the inside of every subdomain, from the tangent at zero
        mixed = torch.from_numpy(mixed).to(self.dev)
        where = [torch.nonzero(self.sub == s) for s in range(self.case["per"] ** 2)]
        lo = torch.stack([w.min(0).values for w in where])
        size = torch.stack([w.max(0).values for w in where]) - lo + 1
        H, W = (size.max(0).values + 1).tolist()
        win = (lo[:, 0], lo[:, 1], H, W)
        tri = (self.at((lo[:, 0], lo[:, 1], H - 1, W - 1), self.sub, -1)
               == torch.arange(len(where), device=self.dev)[:, None, None])[..., None].expand(-1, -1, -1, 2).double()
        inside = self.at(win, self.free & ~mixed, False)
        inside &= ((torch.arange(H, device=self.dev)[None, :, None] <= size[:, 0, None, None])
                   & (torch.arange(W, device=self.dev)[None, None, :] <= size[:, 1, None, None]))
        K = self.cells(win, torch.zeros(len(where), H, W, d, dtype=torch.float64, device=self.dev), tri, True)[1]
        for s in range(len(where)):
            one = (lo[s:s + 1, 0], lo[s:s + 1, 1], H, W)
            edge = P[lo[s, 0]:lo[s, 0] + size[s, 0] + 1, lo[s, 1]:lo[s, 1] + size[s, 1] + 1]
            cols = torch.nonzero(edge.abs().amax((0, 1, 2)) > 0)[:, 0]
            if not len(cols):
                continue
            G = torch.zeros(1, H, W, d, len(cols), dtype=torch.float64, device=self.dev)
            G[0, :edge.shape[0], :edge.shape[1]] = edge[..., cols]
            G *= self.at(one, mixed, False)[..., None, None]
            X = _block_solve(K[s:s + 1], inside[s:s + 1], -_times(K[s:s + 1], G))
            _, j, i = torch.nonzero(inside[s:s + 1], as_tuple=True)
            P[(lo[s, 0] + j)[:, None], (lo[s, 1] + i)[:, None], :, cols[None, :]] = X[0, j, i].transpose(1, 2)
        return P

    def apply(self, K, V):
        """DF V on the free rows, V [nodes y, nodes x, d, m]."""
        parts = [_times(K, V[None, ..., q:q + 64])[0] for q in range(0, V.shape[-1], 64)]
        return torch.cat(parts, -1) * self.free[..., None, None]

    def coarse_matrix(self, P, U):
        K = self.tangent(U)
        flat = P.reshape(-1, P.shape[-1])
        return flat.T @ self.apply(K, P).reshape(flat.shape), K

    def coarse_newton(self, P, U, load, rtol=1e-5, atol=1e-11):
        """T_0(u) of Eq. 9 as its correction P_0 c on the grid, with the stopping rule of the solves."""
        flat = P.reshape(-1, P.shape[-1])
        c = torch.zeros(P.shape[-1], dtype=torch.float64, device=self.dev)
        g = flat.T @ self.residual(U, load).reshape(-1)
        tol = max(atol, rtol * float(g.norm()))
        for _ in range(50):
            if float(g.norm()) <= tol:
                break
            A0, _ = self.coarse_matrix(P, U - (flat @ c).reshape(U.shape))
            s, alpha = torch.linalg.solve(A0, g), 1.0
            for _ in range(10):
                t = flat.T @ self.residual(U - (flat @ (c + alpha * s)).reshape(U.shape), load).reshape(-1)
                if float(t.norm()) <= (1 - 1e-4 * alpha) * float(g.norm()):
                    break
                alpha /= 2
            c, g = c + alpha * s, t
        return (flat @ c).reshape(U.shape)

    def global_newton(self, load_steps):
        U = torch.zeros(self.n + 1, self.n + 1, self.d, dtype=torch.float64, device=self.dev)
        for step in range(1, load_steps + 1):
            for _ in range(30):
                F = self.residual(U, step / load_steps)
                size = float(F.norm())
                if size < (1e-13 if step == load_steps else 1e-6):
                    break
                s = _block_solve(self.tangent(U), self.free[None], F[None, ..., None])[0, ..., 0]
                if not float(s.norm()) > 1e-14 * float(U.norm()):
                    break
                for alpha in (1.0, 0.5, 0.25, 0.125):
                    T = self.residual(U - alpha * s, step / load_steps)
                    if float(T.norm()) < size:
                        break
                if not float(T.norm()) < size:
                    break  # at the rounding floor
                U = U - alpha * s
        return U


def _in_parts(K, mask, rhs):
    """_block_solve on a few windows at a time, to bound the memory of the line blocks."""
    B, H, W, d, m = rhs.shape
    step = max(1, int(4e9 / (8 * 6 * H * (W * d) ** 2)))
    return torch.cat([_block_solve(K[q:q + step], mask[q:q + step], rhs[q:q + step]) for q in range(0, B, step)])


def _network(params, X, sizes):
    """The network on inputs X: tanh-form GELU between its three layers."""
    A, o = X, 0
    for layer, (fi, fo) in enumerate(zip(sizes[:-1], sizes[1:])):
        Wt, o = params[o:o + fi * fo].reshape(fo, fi), o + fi * fo
        A, o = A @ Wt.T + params[o:o + fo], o + fo
        if layer < 2:
            A = 0.5 * A * (1 + torch.tanh(math.sqrt(2 / math.pi) * (A + 0.044715 * A ** 3)))
    return A


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return None  # minibatch training in BF16: 64-bit arithmetic takes another path
    if kind == "infer":
        st = prepare(case, seed)
        net = st["net"]
        params = torch.from_numpy(net.params()).double()
        return _network(params, torch.from_numpy(st["X"]).double(), [net.n_in, net.h1, net.h2, net.n_out])
    n, d = case["n"], _ndof(case)
    if kind == "solve":
        # whole-mesh elimination, one Newton step after another: within seconds up to these sizes
        if n * d > (520 if d == 1 else 260):
            return None
        return _Grid(case, seed).global_newton(case["load_steps"]).reshape(-1)
    grid = _Grid(case, seed)
    U = torch.from_numpy(_state(case, seed)).to(grid.dev).reshape(n + 1, n + 1, d)
    load = _load(case)
    if kind == "residual":
        return grid.residual(U, load).reshape(-1)
    coupling = case["coupling"]
    P0c, x = torch.zeros_like(U), U
    if coupling != "one":
        P = grid.basis()
        P0c = grid.coarse_newton(P, U, load)
        x = U - P0c if coupling == "hybrid" else U
    win, tri, unknown, owned = grid.subdomains()
    w = grid.local_newton(win, tri, unknown, x, load)
    if kind == "corrections":
        Fx = grid.paste(win, owned, grid.at(win, x) - w) + P0c
        return dict(Fx=Fx.reshape(-1), its=None, status=None)
    v = torch.from_numpy(_direction(case, seed)).to(grid.dev).reshape(U.shape)
    w0 = torch.zeros_like(v)
    if coupling != "one":
        A0, K0 = grid.coarse_matrix(P, U - P0c)
        flat = P.reshape(-1, P.shape[-1])
        g = flat.T @ grid.apply(K0, v[..., None]).reshape(-1)
        w0 = (flat @ torch.linalg.solve(A0, g)).reshape(v.shape)
        if coupling == "hybrid":
            v = v - w0
    K = grid.cells(win, w, tri, True)[1]
    q = _times(K, grid.at(win, v)[..., None])
    z = _in_parts(K, unknown, q)[..., 0]
    return (grid.paste(win, owned, z) + w0).reshape(-1)
