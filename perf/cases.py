"""Performance cases: the calls a user of the solver library makes, from the smallest to the largest.

A case names one public call (`call`) on one workload family, with its size, degree and vector type:

  apply     y = A x                               solver.apply
  residual  r = f - A u                           solver.residual
  smooth    one block Gauss-Seidel sweep          solver.smooth
  vcycle    z = M^-1 r, optionally with the       solver.vcycle
            learned boundary-cell correction
  solve     FGMRES(30) to `tol` from x = 0        solver.solve
  forward   MLP inference over boundary cells     mlp.forward
  gradients one MLP training step's gradients     mlp.gradients

`exact` restates the discretisation, the sweep, the V-cycle and the MLP in plain 64-bit torch on full
background grids (class Level); it takes only the problem description from the repository.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_2506_12899_gb300 as sbm
import workloads as W


def listed():
    return [
        # a coarse 2D operator call of an iteration the user drives: nothing but the latency of a call
        dict(name="apply_f64_disk2d_p1_32", call="apply", family="disk2d", n=32, p=1, dtype="f64"),
        # the residual of a fine 2D mesh in the user's own iteration: vectors of 58 MB
        dict(name="residual_f32_star2d_p2_2048", call="residual", family="star2d", n=2048, p=2, dtype="f32"),
        # the operator at the highest 3D order, in a user's own Krylov method
        dict(name="apply_f32_ellipsoid3d_p3_96", call="apply", family="ellipsoid3d", n=96, p=3, dtype="f32"),
        # one post-smoothing (reverse) sweep of a 3D p = 2 level
        dict(name="smooth_f32_sphere3d_p2_112", call="smooth", family="sphere3d", n=112, p=2, dtype="f32", reverse=True),
        # one preconditioner application inside another Krylov method, the benchmark workload
        dict(name="vcycle_f32_star2d_p2_512", call="vcycle", family="star2d", n=512, p=2, dtype="f32", learned=False),
        # the same in 3D at p = 1, a mid-sized mesh whose levels all fit the caches
        dict(name="vcycle_f32_sphere3d_p1_64", call="vcycle", family="sphere3d", n=64, p=1, dtype="f32", learned=False),
        # the plain FP64 preconditioner in 3D
        dict(name="vcycle_f64_sphere3d_p2_64", call="vcycle", family="sphere3d", n=64, p=2, dtype="f64", learned=False),
        # the preconditioner with the learned correction attached, on its 2D family
        dict(name="vcycle_learned_star2d_p3_128", call="vcycle", family="random_star2d", n=128, p=3, dtype="f32", learned=True),
        # inference over the boundary cells of a 96^3 p = 3 mesh
        dict(name="mlp_forward_3d_p3_16384", call="forward", dim=3, p=3, hidden=128, rows=16384),
        # one minibatch of the 3D network's training (the default batch of 4096)
        dict(name="mlp_gradients_3d_p3_4096", call="gradients", dim=3, p=3, hidden=128, rows=4096),
        # the benchmark: one whole solve of the 512^2 p = 2 star
        dict(name="solve_f32_star2d_p2_512", call="solve", family="star2d", n=512, p=2, dtype="f32", tol=1e-8),
        # the largest solve: 96^3 p = 3 ellipsoid, two smoothing steps before and after, to the 1e-12 of the paper
        dict(name="solve_f32_ellipsoid3d_p3_96", call="solve", family="ellipsoid3d", n=96, p=3, dtype="f32", tol=1e-12),
    ]


def draw(rng):
    call = rng.choice(["apply", "residual", "smooth", "vcycle", "vcycle", "solve", "forward", "gradients"])
    if call in ("forward", "gradients"):
        dim, p = rng.choice([2, 3]), rng.choice([1, 2, 3])
        most = 16384 if call == "forward" else 4096
        return dict(call=call, dim=dim, p=p, hidden=rng.choice([32, 64, 96, 128, 128, 200, 256]),
                    rows=int(round(math.exp(rng.uniform(math.log(40), math.log(most))))))
    # meshes of 4..7 times a power of two cells per direction: the coarsest level stays small
    if call == "solve":                             # the families whose solves converge at every size
        family, p = rng.choice([("disk2d", 1), ("star2d", 2), ("random_star2d", 3), ("sphere3d", 1), ("sphere3d", 2),
                                ("ellipsoid3d", 3)])
    else:
        family, p = rng.choice(["disk2d", "star2d", "random_star2d", "sphere3d", "ellipsoid3d"]), rng.choice([1, 2, 2, 3])
    if family.endswith("2d"):
        lo, hi = (32, 512) if call == "solve" else (32, 2048)
    else:
        lo, hi = (16, 48 if p == 3 else 64) if call in ("solve", "vcycle") else (16, 96 if p == 3 else 112)
    sizes = [c << k for c in (4, 5, 6, 7) for k in range(2, 10) if lo <= c << k <= hi]
    case = dict(call=call, family=family, n=rng.choice(sizes), p=p, dtype=rng.choice(["f32", "f32", "f64"]),
                geometry=rng.randrange(5))
    if call == "solve":
        case["tol"] = 1e-12                         # the tolerance of the paper's tables
    if call == "smooth":
        case["reverse"] = rng.random() < 0.5
    if call == "vcycle":
        case["learned"] = p == 3 and rng.random() < 0.5
    if call in ("smooth", "vcycle") and rng.random() < 0.25:
        case["ordering"] = 1                        # red-black instead of the 2^d colours
    return case


# ------------------------------------------------------------------------------------------ inputs
def _problem(case):
    n, p, seed = case["n"], case["p"], case.get("geometry", 0)
    if case["family"] == "disk2d":
        prob = W.disk2d_p1(n, seed) if p == 1 else W.star2d_p2(n, seed).replace(p=p, shape=W.disk(2, seed))
    elif case["family"] == "star2d":
        prob = W.star2d_p2(n, seed).replace(p=p)
    elif case["family"] == "random_star2d":
        prob = W.random_star2d_p3(n, 1000 + seed).replace(p=p)
    elif case["family"] == "sphere3d":
        prob = W.sphere3d(n, p, seed)
    else:
        prob = W.ellipsoid3d_p3(n, seed).replace(p=p, coarsest_n=4, extension=1 if p > 1 else 0)
    return prob.replace(ordering=case.get("ordering", 0))


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(n, dtype, g):
    return 2 * torch.rand(n, dtype=dtype, device="cuda", generator=g) - 1


def _features(dim, p, rows, g):
    """Rows as the library's feature gather makes them: a patch residual of norm 1, shifts d / h on the
    surrogate faces (zero on the others), the volume fraction, the mask of the surrogate faces."""
    np_, nq = (p + 1) ** dim, (p + 1) ** (dim - 1)
    patch = torch.randn(rows, 3 ** dim * np_, device="cuda", generator=g)
    patch /= patch.norm(dim=1, keepdim=True)
    mask = (torch.rand(rows, 2 * dim, device="cuda", generator=g) < 0.3).float()
    shifts = 0.8 * _uniform((rows, 2 * dim, nq * dim), torch.float32, g) * mask[:, :, None]
    kappa = 0.75 + 0.25 * torch.rand(rows, 1, device="cuda", generator=g)
    return torch.cat([patch, shifts.reshape(rows, -1), kappa, mask], dim=1).contiguous()


def _mlp_params(dim, p, hidden, g):
    """He-normal weights and small biases, packed W1 b1 W2 b2 W3 b3 (input-major)."""
    np_ = (p + 1) ** dim
    F = 3 ** dim * np_ + 2 * dim * (p + 1) ** (dim - 1) * dim + 1 + 2 * dim
    parts = []
    for a, b, scale in ((F, hidden, 2.0), (hidden, hidden, 2.0), (hidden, np_, 1.0)):
        parts.append((torch.randn(a, b, device="cuda", generator=g) * math.sqrt(scale / a)).reshape(-1))
        parts.append(0.05 * torch.randn(b, device="cuda", generator=g))
    return torch.cat(parts).cpu().numpy()


def _mlp_inputs(case, seed):
    g = _generator(seed)
    params = _mlp_params(case["dim"], case["p"], case["hidden"], g)
    X = _features(case["dim"], case["p"], case["rows"], g)
    T = torch.randn(case["rows"], (case["p"] + 1) ** case["dim"], device="cuda", generator=g)
    return params, X, T


def _load(rhs, coords, n, np_, seed):
    """Another source term: the manufactured load, each cell's entries scaled by a smooth field."""
    rng = np.random.default_rng(seed)
    k, phase = rng.uniform(1.0, 4.0, 3), rng.uniform(0.0, 2 * math.pi)
    amp = 1.0 + 0.5 * np.sin((coords + 0.5) / n @ k + phase)
    return rhs * torch.from_numpy(np.repeat(amp, np_)).to(rhs.device)


def _correction_scale(case):
    return 0.05                                     # the trained networks' targets have an RMS of this order


def prepare(case, seed):
    call = case["call"]
    if call in ("forward", "gradients"):
        params, X, T = _mlp_inputs(case, seed)
        mlp = sbm.Mlp(case["dim"], case["p"], case["hidden"])
        mlp.set_params(params)
        return dict(call=call, mlp=mlp, X=X, T=T)
    prob = _problem(case)
    solver = sbm.Solver(prob, precision=case["dtype"])
    N, dtype = solver.n_dof(), torch.float32 if case["dtype"] == "f32" else torch.float64
    state = dict(call=call, solver=solver)
    if call == "solve":
        state["tol"] = case["tol"]
        state["b"] = _load(solver.rhs(), solver.layout(), prob.n, (prob.p + 1) ** prob.dim, seed)
        return state
    g = _generator(seed)
    state["x"] = _uniform(N, dtype, g)
    if call in ("residual", "smooth"):
        state["f"] = _uniform(N, dtype, g)
    if call == "smooth":
        state["reverse"] = case["reverse"]
    if call == "vcycle" and case["learned"]:
        mlp = sbm.Mlp(prob.dim, prob.p, 128)
        mlp.set_params(_mlp_params(prob.dim, prob.p, 128, _generator(seed + 1)))
        solver.attach_mlp(mlp, scale=_correction_scale(case))
    return state


def run(state):
    call = state["call"]
    if call == "forward":
        return state["mlp"].forward(state["X"])
    if call == "gradients":
        loss, grad = state["mlp"].gradients(state["X"], state["T"])
        return dict(grad=grad, loss=np.float32(loss))   # the library sums the loss in 32 bits
    solver = state["solver"]
    if call == "apply":
        return solver.apply(state["x"])
    if call == "residual":
        return solver.residual(state["f"], state["x"])
    if call == "smooth":
        return solver.smooth(state["f"], state["x"], reverse=state["reverse"])
    if call == "vcycle":
        return solver.vcycle(state["x"])
    x = torch.zeros_like(state["b"])
    solver.solve(state["b"], x, tol=state["tol"])
    return x


# -------------------------------------------------------------------------------------------- work
def _volume(prob):
    s = prob.shape
    if s.kind == W.SHAPE_STAR:
        return math.pi * s.radius ** 2 * (1 + 0.5 * s.amp ** 2)
    if s.kind == W.SHAPE_ELLIPSOID:
        return 4 / 3 * math.pi * s.semi[0] * s.semi[1] * s.semi[2]
    return math.pi * s.radius ** 2 if prob.dim == 2 else 4 / 3 * math.pi * s.radius ** 3


def work(case):
    call = case["call"]
    if call in ("forward", "gradients"):
        p, dim, H, R = case["p"], case["dim"], case["hidden"], case["rows"]
        O = (p + 1) ** dim
        F = 3 ** dim * O + 2 * dim * (p + 1) ** (dim - 1) * dim + 1 + 2 * dim
        params = F * H + H * H + H * O
        if call == "forward":
            return dict(bytes=4 * (R * (F + O) + params), flops=2 * R * params)
        return dict(bytes=4 * (R * (F + O) + 2 * params), flops=2 * R * (3 * params - F * H))
    prob = _problem(case)
    w, dim, n1 = (4 if case["dtype"] == "f32" else 8), prob.dim, prob.p + 1
    cells = _volume(prob) * (prob.n / (prob.hi[0] - prob.lo[0])) ** dim
    N = cells * n1 ** dim
    boundary = 2.5 * dim * cells ** ((dim - 1) / dim)   # cells with a surrogate face, roughly
    inverses = w * boundary * n1 ** (2 * dim)
    apply_flops = N * dim * (6 * n1 + 2)            # self and two neighbours' 1D matrices per direction
    sweep_flops = N * dim * (8 * n1 + 2)            # neighbours, then the fast diagonalisation
    if call == "apply":
        return dict(bytes=2 * w * N, flops=apply_flops)
    if call == "residual":
        return dict(bytes=3 * w * N, flops=apply_flops)
    if call == "smooth":
        return dict(bytes=3 * w * N + inverses, flops=sweep_flops)
    # every level of the hierarchy once in each sweep, residual and transfer
    below = sum((q / n1) ** dim for q in range(2, n1)) + (2 / n1) ** dim / (2 ** dim - 1)
    cycle_flops = (1 + below) * ((prob.pre_smooth + prob.post_smooth) * sweep_flops + apply_flops)
    if call == "vcycle":
        return dict(bytes=2 * w * N + inverses, flops=cycle_flops)
    steps = 27 if case["tol"] > 1e-9 else 50        # about what the listed solves take
    basis = 2 * 8 * N * min(steps, 30) / 2          # two projections over half the basis on average, FP64-sized
    return dict(bytes=16 * N + steps * (inverses + basis), flops=steps * (cycle_flops + apply_flops + 4 * N * steps))


# ------------------------------------------------------------------------------------------- exact
F64 = dict(dtype=torch.float64, device="cuda")


def _lagrange(nodes, y):
    """Values of the Lagrange basis on `nodes` at y (any shape): shape y.shape + (len(nodes),)."""
    cols = []
    for k, xk in enumerate(nodes):
        v = torch.ones_like(y)
        for j, xj in enumerate(nodes):
            if j != k:
                v = v * (y - xj) / (xk - xj)
        cols.append(v)
    return torch.stack(cols, dim=-1)


def _lagrange_derivative(nodes, y):
    cols = []
    for k, xk in enumerate(nodes):
        d = torch.zeros_like(y)
        for i, xi in enumerate(nodes):
            if i == k:
                continue
            term = torch.full_like(y, 1 / (xk - xi))
            for j, xj in enumerate(nodes):
                if j != k and j != i:
                    term = term * (y - xj) / (xk - xj)
            d = d + term
        cols.append(d)
    return torch.stack(cols, dim=-1)


def _phi(prob, x):
    """Level set at the points x = [x_0, x_1, ...] (broadcastable tensors)."""
    s = prob.shape
    y = [x[k] - s.center[k] for k in range(prob.dim)]
    if s.kind == W.SHAPE_STAR:
        return torch.sqrt(y[0] ** 2 + y[1] ** 2) - s.radius * (1 + s.amp * torch.sin(s.freq * torch.atan2(y[1], y[0]) + s.phase))
    if s.kind == W.SHAPE_ELLIPSOID:
        q = [sum(s.rot[3 * r + i] * y[r] for r in range(3)) / s.semi[i] for i in range(3)]
        return torch.sqrt(q[0] ** 2 + q[1] ** 2 + q[2] ** 2) - 1
    return torch.sqrt(sum(v ** 2 for v in y)) - s.radius


def _closest(prob, X):
    """Closest points of the boundary {phi = 0} to the points X (m, dim)."""
    s, c = prob.shape, torch.tensor(prob.shape.center[:prob.dim], **F64)
    if s.kind == W.SHAPE_STAR:
        def curve(t):
            r, r1 = s.radius * (1 + s.amp * torch.sin(s.freq * t + s.phase)), s.radius * s.amp * s.freq * torch.cos(s.freq * t + s.phase)
            r2 = -s.radius * s.amp * s.freq ** 2 * torch.sin(s.freq * t + s.phase)
            e, n = torch.stack([torch.cos(t), torch.sin(t)], -1), torch.stack([-torch.sin(t), torch.cos(t)], -1)
            r, r1, r2 = r[..., None], r1[..., None], r2[..., None]
            return c + r * e, r1 * e + r * n, (r2 - r) * e + 2 * r1 * n
        t0 = torch.arange(4096, **F64) * (2 * math.pi / 4096)
        t = torch.cat([t0[torch.cdist(x, curve(t0)[0]).argmin(1)] for x in X.split(20000)])
        for _ in range(30):                         # Newton on (P(t) - x) . P'(t) = 0
            P, P1, P2 = curve(t)
            t = t - ((P - X) * P1).sum(-1) / ((P1 * P1).sum(-1) + ((P - X) * P2).sum(-1))
        return curve(t)[0]
    if s.kind == W.SHAPE_ELLIPSOID:
        R, a = torch.tensor(s.rot, **F64).reshape(3, 3), torch.tensor(s.semi, **F64)
        y = (X - c) @ R
        lo = -a.min() ** 2 + a.min() * y[:, a.argmin()].abs()   # sum (a y / (t + a^2))^2 = 1, decreasing in t
        hi = a.max() * y.norm(dim=1)
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            out = ((a * y / (mid[:, None] + a ** 2)) ** 2).sum(1) > 1
            lo, hi = torch.where(out, mid, lo), torch.where(out, hi, mid)
        t = (0.5 * (lo + hi))[:, None]
        return c + (a ** 2 * y / (t + a ** 2)) @ R.T
    d = X - c
    return c + s.radius * d / d.norm(dim=1, keepdim=True)


class Level:
    """One level on the full background grid, in 64 bits.  A vector is a tensor of shape
    (n,) * dim + (n1,) * dim (cell axes, then node axes, each with x last); inactive cells are zero."""

    def __init__(self, prob, n, p):
        self.prob, self.n, self.p, self.dim, self.n1 = prob, n, p, prob.dim, p + 1
        d, n1 = self.dim, self.n1
        self.h = (prob.hi[0] - prob.lo[0]) / n
        self.omega = prob.omega_p3 if p == 3 else prob.omega
        x, w = np.polynomial.legendre.leggauss(n1)
        self.x, self.w = torch.tensor(0.5 * (x + 1), **F64), torch.tensor(0.5 * w, **F64)
        ends = torch.tensor([0.0, 1.0], **F64)
        self.e, self.d1 = _lagrange(self.x, ends), _lagrange_derivative(self.x, ends)   # [side][node]
        self.Dm = _lagrange_derivative(self.x, self.x)
        K = self.Dm.T @ torch.diag(self.w) @ self.Dm
        (e0, e1), (d0, d1), s = self.e, self.d1, prob.sigma_face_c * n1 ** 2
        o = torch.outer
        self.K = K                                  # interior penalty halves (rows: test, columns: trial)
        self.Bmm = -0.5 * (o(e1, d1) + o(d1, e1)) + s * o(e1, e1)
        self.Bpp = 0.5 * (o(e0, d0) + o(d0, e0)) + s * o(e0, e0)
        self.Bmp = -0.5 * o(e1, d0) + 0.5 * o(d1, e0) - s * o(e1, e0)
        self.Bpm = 0.5 * o(e0, d1) - 0.5 * o(d0, e1) - s * o(e0, e1)
        self.kappa = self._volume_fractions()
        self.active = self.kappa >= prob.lam if prob.lam_inclusive else self.kappa > prob.lam
        self._order()
        self._faces()
        self._inverses = None

    def _volume_fractions(self):
        prob, n, d, s = self.prob, self.n, self.dim, self.prob.samples
        pts = [prob.lo[k] + self.h * (torch.arange(n, **F64)[:, None] + ((torch.arange(s, **F64) + 0.5) / s)).reshape(-1) for k in range(d)]
        out, rows = [], max(1, int(2e7 / (n * s) ** (d - 1) / s))
        for i in range(0, n, rows):                 # slabs along the slowest direction
            slab = pts[d - 1][i * s:(i + rows) * s]
            grid = [pts[0], pts[1][:, None], None] if d == 3 else [pts[0], None]
            grid[d - 1] = slab.reshape((-1,) + (1,) * (d - 1))
            inside = (_phi(prob, grid) < 0).double()
            shape = [v for m in [len(slab) // s] + [n] * (d - 1) for v in (m, s)]
            out.append(inside.reshape(shape).sum(dim=tuple(range(1, 2 * d, 2))))
        return torch.cat(out) / s ** d

    def _shifted(self, U, dim_, side):
        """The values of the neighbour across face (dim_, side), zero outside the grid."""
        ax = self.dim - 1 - dim_
        V = torch.zeros_like(U)
        src, dst = [slice(None)] * U.dim(), [slice(None)] * U.dim()
        src[ax], dst[ax] = (slice(1, None), slice(None, -1)) if side else (slice(None, -1), slice(1, None))
        V[tuple(dst)] = U[tuple(src)]
        return V

    def _order(self):
        """The compact order: by colour; within one, cells with a surrogate face first, by their set of
        such faces; then by background index."""
        d, n = self.dim, self.n
        self.present = [[self._shifted(self.active, k, s) & self.active for s in (0, 1)] for k in range(d)]
        act = self.active.reshape(-1)
        mask = sum((~self.present[k][s]).reshape(-1).long() << (2 * k + s) for k in range(d) for s in (0, 1))
        lin = torch.arange(n ** d, device="cuda")
        colour = sum((lin // n ** k % n % 2) << k for k in range(d))
        key = ((colour * 2 + (mask == 0)) * 2 ** (2 * d) + mask) * n ** d + lin
        lin = lin[act]
        self.order = lin[key[act].argsort()]
        self.colour, self.boundary = colour, self.order[mask[self.order] > 0]

    def grid(self, v):
        U = torch.zeros(self.n ** self.dim, self.n1 ** self.dim, **F64)
        U[self.order] = v.reshape(len(self.order), -1).double()
        return U.reshape((self.n,) * self.dim + (self.n1,) * self.dim)

    def cells(self, U):
        return U.reshape(self.n ** self.dim, -1)

    def compact(self, U):
        return self.cells(U)[self.order].reshape(-1)

    def along(self, M, U, k):
        """The matrix M on the nodes of direction k."""
        ax = U.dim() - 1 - k
        return (U.movedim(ax, -1) @ M.T).movedim(-1, ax)

    def _tensor(self, mats):
        """The matrix of a tensor product, mats[k] acting in direction k (x fastest)."""
        out = mats[0]
        for M in mats[1:]:
            out = torch.kron(M, out)
        return out

    def _faces(self):
        """Surrogate faces: cells, trace T, normal derivative G and extended value E as matrices on the
        cell's values, quadrature weights."""
        d, n, n1 = self.dim, self.n, self.n1
        eye, self.faces = torch.eye(n1, **F64), []
        for k, side in itertools.product(range(d), (0, 1)):
            cell = (self.active & ~self.present[k][side]).reshape(-1).nonzero()[:, 0]
            tang = [m for m in range(d) if m != k]
            T = self._tensor([self.e[side][None] if m == k else eye for m in range(d)])
            G = self._tensor([self.d1[side][None] if m == k else eye for m in range(d)])
            wq = self._tensor([self.w[:, None]] * (d - 1))[:, 0]
            ref = torch.zeros(n1 ** (d - 1), d, **F64)
            ref[:, k] = side
            for q, m in enumerate(tang):
                ref[:, m] = self.x[(torch.arange(n1 ** (d - 1), device="cuda") // n1 ** q) % n1]
            idx = torch.stack([cell // n ** m % n for m in range(d)], 1)
            X = torch.tensor(self.prob.lo[:d], **F64) + self.h * (idx[:, None, :] + ref)
            dh = (_closest(self.prob, X.reshape(-1, d)).reshape(X.shape) - X) / self.h if len(cell) else torch.zeros_like(X)
            if self.prob.extension == 0:
                E = T + dh[:, :, k, None] * G
                for m in tang:
                    E = E + dh[:, :, m, None] * (self._tensor([self.Dm if q == m else eye for q in tang]) @ T)
            else:
                E = torch.ones(len(cell), len(ref), 1, **F64)
                for m in range(d):                  # x fastest: the later directions go in front
                    E = (_lagrange(self.x, ref[:, m] + dh[:, :, m])[..., :, None] * E[..., None, :]).flatten(2)
            self.faces.append((cell, k, side, T, G, E, wq, dh))

    def _face_matrix(self, face):
        """The lift of (normal derivative, extended value) to the cell's test functions: y = A G u + B E u."""
        _, _, side, T, G, _, wq, _ = face
        sg, sigma = (1.0 if side else -1.0), self.prob.sigma_bnd_c * self.n1 ** 2
        return -sg * T.T * wq, sigma * T.T * wq - self.prob.alpha * sg * G.T * wq

    def apply(self, U):
        U = U.contiguous()
        Y = torch.zeros(U.shape, **F64)
        for k in range(self.dim):
            lo, hi = ((self.present[k][s].reshape(self.present[k][s].shape + (1,) * self.dim)).double() for s in (0, 1))
            s = self.along(self.K, U, k) + lo * self.along(self.Bpp, U, k) + hi * self.along(self.Bmm, U, k)
            s += self.along(self.Bpm, self._shifted(U, k, 0), k) + self.along(self.Bmp, self._shifted(U, k, 1), k)
            for m in range(self.dim):
                if m != k:
                    s *= self.w.reshape((-1,) + (1,) * m)
            Y += s
        y, u = self.cells(Y), self.cells(U)
        for face in self.faces:
            cell, G, E = face[0], face[4], face[5]
            A, B = self._face_matrix(face)
            uk = u[cell]
            y.index_add_(0, cell, uk @ G.T @ A.T + torch.bmm(E, uk[:, :, None])[:, :, 0] @ B.T)
        y *= self.active.reshape(-1, 1)
        return Y * self.h ** (self.dim - 2)

    def inverses(self):
        """(inverse of the interior block, slot of each cell among the boundary blocks, their inverses)."""
        if self._inverses is None:
            d, eye = self.dim, torch.diag(self.w)
            blocks = torch.zeros(len(self.boundary) + 1, self.n1 ** d, self.n1 ** d, **F64)
            slot = torch.full((self.n ** d,), len(self.boundary), device="cuda")
            slot[self.boundary] = torch.arange(len(self.boundary), device="cuda")
            for k in range(d):
                dense = lambda M: self._tensor([M if m == k else eye for m in range(d)])  # noqa: E731
                blocks += dense(self.K)
                for s, B in ((0, self.Bpp), (1, self.Bmm)):
                    here = torch.cat([self.present[k][s].reshape(-1)[self.boundary], torch.ones(1, dtype=torch.bool, device="cuda")])
                    blocks[here] += dense(B)
            for face in self.faces:
                A, B = self._face_matrix(face)
                blocks.index_add_(0, slot[face[0]], A @ face[4] + B @ face[5])
            self._inverses = slot, torch.linalg.inv(blocks * self.h ** (d - 2))
        return self._inverses

    def sweep(self, F, U, reverse):
        """One block Gauss-Seidel sweep, colour by colour (red-black: by the parity of the index sum)."""
        slot, inv = self.inverses()
        key, U = self.colour, U.contiguous()
        if self.prob.ordering == 1:
            key = sum((self.colour >> k) & 1 for k in range(self.dim)) % 2
        for c in range(int(key.max()) + 1)[::-1 if reverse else 1]:
            cell = self.order[key[self.order] == c]
            r = self.cells(F - self.apply(U))[cell]
            interior = slot[cell] == len(inv) - 1
            z = r @ inv[-1].T
            z[~interior] = torch.bmm(inv[slot[cell[~interior]]], r[~interior][:, :, None])[:, :, 0]
            self.cells(U)[cell] += self.omega * z
        return U

    def prolong(self, Ec, coarse):
        for k in range(self.dim):
            if coarse.n == self.n:
                Ec = self.along(_lagrange(coarse.x, self.x), Ec, k)
            else:
                ax = self.dim - 1 - k
                Ec = torch.stack([self.along(_lagrange(coarse.x, 0.5 * (o + self.x)), Ec, k) for o in (0, 1)], ax + 1).flatten(ax, ax + 1)
        return Ec * self.active.reshape(self.active.shape + (1,) * self.dim)

    def restrict(self, R, coarse):
        for k in range(self.dim):
            if coarse.n == self.n:
                R = self.along(_lagrange(coarse.x, self.x).T, R, k)
            else:
                ax = self.dim - 1 - k
                R = sum(self.along(_lagrange(coarse.x, 0.5 * (o + self.x)).T, R.unflatten(ax, (-1, 2)).select(ax + 1, o), k) for o in (0, 1))
        return R * coarse.active.reshape(coarse.active.shape + (1,) * self.dim)


def _levels(prob):
    ns = [prob.n]
    while ns[-1] % 2 == 0 and ns[-1] // 2 >= prob.coarsest_n:
        ns.append(ns[-1] // 2)
    levels = [Level(prob, n, 1) for n in ns[::-1]] + [Level(prob, prob.n, q) for q in range(2, prob.p + 1)]
    empty = [i for i, L in enumerate(levels) if not len(L.order)]
    return levels[empty[-1] + 1:] if empty else levels


def _vcycle(levels, R, correct=None):
    L, prob = levels[-1], levels[-1].prob
    if len(levels) == 1:
        N = len(L.order) * L.n1 ** L.dim
        A = torch.stack([L.compact(L.apply(L.grid(v))) for v in torch.eye(N, **F64)], 1)
        return L.grid(torch.linalg.solve(A, L.compact(R)))
    Z = torch.zeros_like(R)
    for _ in range(prob.pre_smooth):
        Z = L.sweep(R, Z, False)
    coarse = levels[-2]
    Z = Z + L.prolong(_vcycle(levels[:-1], L.restrict(R - L.apply(Z), coarse)), coarse)
    for _ in range(prob.post_smooth):
        Z = L.sweep(R, Z, True)
    return correct(L, R, Z) if correct else Z


def _mlp(dim, p, hidden, params):
    """The layers (W, b) of a packed parameter vector."""
    np_ = (p + 1) ** dim
    F = 3 ** dim * np_ + 2 * dim * (p + 1) ** (dim - 1) * dim + 1 + 2 * dim
    v, out, at = torch.tensor(params, **F64), [], 0
    for a, b in ((F, hidden), (hidden, hidden), (hidden, np_)):
        out.append((v[at:at + a * b].reshape(a, b), v[at + a * b:at + a * b + b]))
        at += a * b + b
    return out


def _forward(layers, X):
    acts = [X]
    for i, (Wt, b) in enumerate(layers):
        z = acts[-1] @ Wt + b
        acts.append(z.clamp(min=0) if i < 2 else z)
    return acts


def _corrected(L, R, Z, layers, scale):
    """The learned correction of the boundary cells (features, MLP, scatter)."""
    d, n, n1, m = L.dim, L.n, L.n1, len(L.boundary)
    nq = n1 ** (d - 1)
    res = torch.cat([L.cells(R - L.apply(Z)), torch.zeros(1, n1 ** d, **F64)])   # the last row: no such cell
    idx = torch.stack([L.boundary // n ** k % n for k in range(d)], 1)
    patch = []
    for o in range(3 ** d):
        j = idx + torch.tensor([o // 3 ** k % 3 - 1 for k in range(d)], device="cuda")
        lin = sum(j[:, k] * n ** k for k in range(d))
        patch.append(res[torch.where(((j >= 0) & (j < n)).all(1), lin, torch.full_like(lin, n ** d))])
    patch = torch.cat(patch, 1)
    s = patch.norm(dim=1, keepdim=True)
    s = torch.where(s > 0, s, torch.ones_like(s))
    at = torch.full((n ** d,), -1, device="cuda")
    at[L.boundary] = torch.arange(m, device="cuda")
    shifts, mask = torch.zeros(m, 2 * d, nq, d, **F64), torch.zeros(m, 2 * d, **F64)
    for cell, k, side, _, _, _, _, dh in L.faces:
        shifts[at[cell], 2 * k + side] = dh
        mask[at[cell], 2 * k + side] = 1
    X = torch.cat([patch / s, shifts.reshape(m, -1), L.kappa.reshape(-1)[L.boundary][:, None], mask], 1)
    Z = Z.contiguous().clone()
    L.cells(Z)[L.boundary] += scale * s * L.h ** (2 - d) * _forward(layers, X)[-1]
    return Z


def exact(case, seed):
    call = case["call"]
    if call == "solve":
        return None                                 # an iterate at a tolerance, not a computed number
    if call in ("forward", "gradients"):
        params, X, T = _mlp_inputs(case, seed)
        layers = _mlp(case["dim"], case["p"], case["hidden"], params)
        acts = _forward(layers, X.double())
        if call == "forward":
            return acts[-1]
        err = acts[-1] - T.double()
        grads, dZ = [], 2 * err / err.numel()
        for i in (2, 1, 0):
            grads = [(acts[i].T @ dZ).reshape(-1), dZ.sum(0)] + grads
            dZ = (dZ @ layers[i][0].T) * (acts[i] > 0) if i else None
        return dict(grad=torch.cat(grads), loss=(err ** 2).mean())
    prob = _problem(case)
    L = Level(prob, prob.n, prob.p) if call != "vcycle" else None
    levels = _levels(prob) if call == "vcycle" else [L]
    L = levels[-1]
    N, g = len(L.order) * L.n1 ** L.dim, _generator(seed)
    dtype = torch.float32 if case["dtype"] == "f32" else torch.float64
    U = L.grid(_uniform(N, dtype, g))
    if call == "vcycle":
        correct = None
        if case["learned"]:
            layers = _mlp(prob.dim, prob.p, 128, _mlp_params(prob.dim, prob.p, 128, _generator(seed + 1)))
            correct = lambda L, R, Z: _corrected(L, R, Z, layers, _correction_scale(case))  # noqa: E731
        return L.compact(_vcycle(levels, U, correct))
    if call == "apply":
        return L.compact(L.apply(U))
    F = L.grid(_uniform(N, dtype, g))
    return L.compact(F - L.apply(U)) if call == "residual" else L.compact(L.sweep(F, U, case["reverse"]))
