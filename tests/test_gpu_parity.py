"""Parity of the CUDA path (through the C-ABI binding) with the CPU FP64 oracle.

Every comparison maps the library's compact, colour-major layout onto the oracle's natural
ordering with the layout the library reports, then compares element by element.  FP64
tolerances: 1e-12 relative for the operator and the transfers; for operations that apply
cell-block inverses (smoother, V-cycle) max(1e-12, n_p eps cond(A_KK)) (see `block_tol`);
1e-10 relative L2 for FGMRES solutions with equal iteration counts.  FP32 tolerances are derived from the
FP32 unit roundoff (6e-8) times the operation's amplification (stated per test).
"""
import zlib

import numpy as np
import pytest

import workloads as W
from oracle import krylov as K
from oracle import multigrid as MG

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


from _pairs import Pair, _dof_map  # noqa: E402,F401


CASES = {
    "disk2d_p1_n32": W.disk2d_p1(32, 0),
    "disk2d_p1_n32_s3": W.disk2d_p1(32, 3),
    "star2d_p2_n32": W.star2d_p2(32, 1),
    "star2d_p3_n16": W.star2d_p2(16, 2).replace(p=3),
    "sphere3d_p1_n8": W.sphere3d(8, 1, 2),
    "sphere3d_p2_n8": W.sphere3d(8, 2, 3),
    "ellipsoid3d_p3_n12": W.ellipsoid3d_p3(12, 4),
    "disk2d_p2_poly": W.disk2d_p1(16, 5).replace(p=2, extension=1),
    "box2d_p2": W.Problem(dim=2, n=16, p=2, shape=W.box(0.5)),
    "star2d_p3_n16_ssor": W.star2d_p2(16, 2).replace(p=3, ssor_each=1),
    "complex2d_p1_l3": W.paper_complex2d(3, 1, 0.5),
    "complex2d_p2_l2": W.paper_complex2d(2, 2, 0.75),
    "complex2d_p3_l2": W.paper_complex2d(2, 3, 0.5),
    "paper_disk_p2_l3": W.paper_disk(3, 2, 0.5),
    # smoother and formulation variants (Sec. 2.1, Sec. 3.1, Sec. 5.3)
    "star2d_p2_n32_redblack": W.star2d_p2(32, 1).replace(ordering=1),
    "sphere3d_p2_n8_redblack": W.sphere3d(8, 2, 3).replace(ordering=1),
    "disk2d_p1_n32_jacobi": W.disk2d_p1(32, 0).replace(smoother=1, omega=0.7),
    "ellipsoid3d_p3_n12_jacobi": W.ellipsoid3d_p3(12, 4).replace(smoother=1, omega=0.7, omega_p3=0.6),
    "star2d_p3_n16_chebyshev": W.star2d_p2(16, 2).replace(p=3, smoother=2),
    "sphere3d_p1_n8_chebyshev": W.sphere3d(8, 1, 2).replace(smoother=2, cheb_degree=3),
    "disk2d_p2_penalty_free": W.disk2d_p1(16, 5).replace(p=2, extension=1, alpha=-1.0, sigma_bnd_c=0.0),
}
_pairs = {}


def pair(name, precision="f64", tail=0, cell=0, basis=0):
    """tail: CTAs of the launch that runs the small p = 1 levels' V-cycle (16: a thread-block
    cluster, 1: one CTA, 0: one launch per phase); cell: thread-per-cell kernels (0: size-based
    default, 1: always where (p+1)^d <= 16, -1: never); basis: FGMRES basis storage (0
    double-float, 1 FP64)."""
    key = (name, precision, tail, cell, basis)
    if key not in _pairs:
        _pairs[key] = Pair(CASES[name], precision, 40000 if tail else -1, cell, krylov_basis=basis,
                           tail_cluster_ctas=tail)
    return _pairs[key]


def rel_max(a, b):
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def block_tol(levels):
    """FP64 tolerance for operations that apply cell-block inverses: the rounding error of a
    block solve grows like n_p * eps * cond(A_KK); floor 1e-12."""
    kap = max(np.linalg.cond(lev.disc.diag).max() for lev in levels)
    nb = max(lev.nb for lev in levels)
    return max(1e-12, nb * 2.2e-16 * kap)


@pytest.mark.parametrize("name", list(CASES))
def test_apply_matches_assembled_matrix(name):
    """a1: y = A_l x on every level equals the oracle's assembled CSR product (Eq. 11)."""
    P = pair(name)
    for l, lev in enumerate(P.H.levels):
        x = W.random_vector(lev.N, 11 + l)
        yo = lev.A @ x
        y64 = P.to_oracle(P.gpu.apply(P.to_gpu(x, l), level=l), l)
        assert rel_max(y64, yo) <= 1e-12, (l, rel_max(y64, yo))
        y32 = P.to_oracle(P.gpu.apply(P.to_gpu(x, l, torch.float32), level=l), l)
        # FP32: inputs rounded (6e-8) and ~3d(p+1) terms per entry, entries up to ~|A||x|
        scale = np.abs(abs(lev.A) @ np.abs(x)).max()
        assert np.abs(y32 - yo).max() <= 2e-6 * scale, (l, np.abs(y32 - yo).max() / scale)


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "ellipsoid3d_p3_n12", "star2d_p3_n16"])
def test_apply_unit_columns_tiny(name):
    """Column-by-column equality with the CSR on the coarsest level (every face type present)."""
    P = pair(name)
    lev = P.H.levels[0]
    A = lev.A.toarray()
    for j in range(0, lev.N, max(1, lev.N // 40)):
        e = np.zeros(lev.N)
        e[j] = 1.0
        y = P.to_oracle(P.gpu.apply(P.to_gpu(e, 0), level=0), 0)
        assert np.abs(y - A[:, j]).max() <= 1e-12 * np.abs(A).max()


@pytest.mark.parametrize("cell", [1, -1], ids=["thread_per_cell", "thread_per_dof"])
@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p2_n32", "star2d_p3_n16", "sphere3d_p1_n8", "sphere3d_p2_n8",
                                  "ellipsoid3d_p3_n12"])
def test_kernel_variants(name, cell):
    """Both kernel families (one thread per cell, one thread per dof) for the operator, the
    smoother and the V-cycle, in FP64 and FP32, against the oracle (3D p = 2: the FP32 operator
    and the residual + restriction of the V-cycle one thread per cell, the FP32 smoother one thread
    per line of a cell; 3D p = 3: the FP32 operator and smoother one thread per line; against
    thread per DoF)."""
    P = pair(name, cell=cell)
    L = len(P.H.levels) - 1
    lev = P.H.finest
    x = W.random_vector(lev.N, 3)
    assert rel_max(P.to_oracle(P.gpu.apply(P.to_gpu(x, L)), L), lev.A @ x) <= 1e-12
    scale = np.abs(abs(lev.A) @ np.abs(x)).max()
    y32 = P.to_oracle(P.gpu.apply(P.to_gpu(x, L, torch.float32)), L)
    assert np.abs(y32 - lev.A @ x).max() <= 2e-6 * scale
    f, u0 = W.random_vector(lev.N, 4), W.random_vector(lev.N, 5)
    uo = lev.coloured_sweep(u0.copy(), f)
    ug = P.to_oracle(P.gpu.smooth(P.to_gpu(f, L), P.to_gpu(u0, L)), L)
    assert rel_max(ug, uo) <= block_tol([lev])
    ug32 = P.to_oracle(P.gpu.smooth(P.to_gpu(f, L, torch.float32), P.to_gpu(u0, L, torch.float32)), L)
    assert rel_max(ug32, uo) <= 2e-4
    zo = P.H.vcycle(f)
    z = P.to_oracle(P.gpu.vcycle(P.to_gpu(f, L)), L)
    assert np.linalg.norm(z - zo) <= block_tol(P.H.levels[1:] or P.H.levels) * np.linalg.norm(zo)
    z32 = P.to_oracle(P.gpu.vcycle(P.to_gpu(f, L, torch.float32)), L)
    assert np.linalg.norm(z32 - zo) <= 1e-4 * np.linalg.norm(zo)


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "sphere3d_p2_n8", "ellipsoid3d_p3_n12"])
def test_residual(name):
    P = pair(name)
    lev = P.H.finest
    L = len(P.H.levels) - 1
    f, u = W.random_vector(lev.N, 1), W.random_vector(lev.N, 2)
    r = P.to_oracle(P.gpu.residual(P.to_gpu(f, L), P.to_gpu(u, L)), L)
    ro = f - lev.A @ u
    assert rel_max(r, ro) <= 1e-12


@pytest.mark.parametrize("name", list(CASES))
def test_coloured_smoother_sweep(name):
    """a2: one forward and one reverse coloured block Gauss-Seidel sweep (Eqs. 14, 16)."""
    P = pair(name)
    for l in range(1, len(P.H.levels)):
        lev = P.H.levels[l]
        f, u0 = W.random_vector(lev.N, 3 + l), W.random_vector(lev.N, 5 + l)
        for reverse in (False, True):
            uo = lev.coloured_sweep(u0.copy(), f, reverse=reverse)
            ug = P.gpu.smooth(P.to_gpu(f, l), P.to_gpu(u0, l), level=l, reverse=reverse)
            tol = block_tol([lev])
            assert rel_max(P.to_oracle(ug, l), uo) <= tol, (l, reverse, rel_max(P.to_oracle(ug, l), uo), tol)
            ug32 = P.gpu.smooth(P.to_gpu(f, l, torch.float32), P.to_gpu(u0, l, torch.float32), level=l,
                                reverse=reverse)
            # FP32: rounded inputs and block inverses amplified by cond(A_KK) (<= ~1e3 here)
            assert rel_max(P.to_oracle(ug32, l), uo) <= 2e-4, (l, reverse, rel_max(P.to_oracle(ug32, l), uo))


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p3_n16", "sphere3d_p2_n8", "ellipsoid3d_p3_n12"])
def test_transfers(name):
    """a3/a4: restriction = P^T (Eq. 18) and prolongation P (Eq. 17), masked to active cells."""
    P = pair(name)
    for l in range(1, len(P.H.levels)):
        Pm = P.H.P[l]
        rf = W.random_vector(P.H.levels[l].N, l)
        rc = P.to_oracle(P.gpu.restrict(P.to_gpu(rf, l), level=l), l - 1)
        assert rel_max(rc, Pm.T @ rf) <= 1e-13
        ec, uf = W.random_vector(P.H.levels[l - 1].N, 7 + l), W.random_vector(P.H.levels[l].N, 9 + l)
        out = P.to_oracle(P.gpu.prolong_add(P.to_gpu(ec, l - 1), P.to_gpu(uf, l), level=l), l)
        assert rel_max(out, uf + Pm @ ec) <= 1e-13


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p2_n32", "sphere3d_p1_n8", "ellipsoid3d_p3_n12"])
def test_coarse_solve(name):
    """a5: dense FP64 coarse solve equals the oracle's LU solve."""
    P = pair(name)
    lev = P.H.levels[0]
    r = W.random_vector(lev.N, 4)
    x = np.linalg.solve(lev.A.toarray(), r)
    e = P.to_oracle(P.gpu.coarse_solve(P.to_gpu(r, 0)), 0)
    assert rel_max(e, x) <= 1e-11


@pytest.mark.parametrize("tail", [16, 1, 0], ids=["cluster_tail", "cta_tail", "per_level_launches"])
@pytest.mark.parametrize("name", list(CASES))
def test_vcycle(name, tail):
    """One V-cycle (Sec. 3) equals the oracle's; FP32 V-cycle within its rounding bound.  Run with
    the small p = 1 levels in one thread-block-cluster launch, in one one-CTA launch, and with one
    launch per phase."""
    P = pair(name, tail=tail)
    L = len(P.H.levels) - 1
    r = W.random_vector(P.H.finest.N, 21)
    zo = P.H.vcycle(r)
    z = P.to_oracle(P.gpu.vcycle(P.to_gpu(r, L)), L)
    tol = block_tol(P.H.levels[1:] or P.H.levels)
    assert np.linalg.norm(z - zo) <= tol * np.linalg.norm(zo), (np.linalg.norm(z - zo) / np.linalg.norm(zo), tol)
    z32 = P.to_oracle(P.gpu.vcycle(P.to_gpu(r, L, torch.float32)), L)
    assert np.linalg.norm(z32 - zo) <= 1e-4 * np.linalg.norm(zo), np.linalg.norm(z32 - zo) / np.linalg.norm(zo)


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "disk2d_p1_n32_s3", "star2d_p2_n32", "sphere3d_p1_n8",
                                  "sphere3d_p2_n8", "box2d_p2", "star2d_p3_n16_ssor", "complex2d_p1_l3",
                                  "complex2d_p2_l2", "complex2d_p3_l2", "paper_disk_p2_l3", "star2d_p2_n32_redblack",
                                  "sphere3d_p2_n8_redblack", "disk2d_p1_n32_jacobi", "ellipsoid3d_p3_n12_jacobi",
                                  "star2d_p3_n16_chebyshev", "sphere3d_p1_n8_chebyshev", "disk2d_p2_penalty_free"])
def test_fgmres_fp64_matches_oracle(name):
    """a6: FP64 FGMRES(30) + FP64 V-cycle: same iteration count as the oracle and the solution
    within 1e-10 relative L2."""
    P = pair(name)
    F = P.H.finest
    L = len(P.H.levels) - 1
    bo = F.disc.rhs()
    xo, oi = K.fgmres(lambda v: F.A @ v, P.H.vcycle, bo, tol=1e-8, m=30, max_it=300)
    b = P.gpu.rhs()
    assert rel_max(P.to_oracle(b, L), bo) <= 1e-13
    x = torch.zeros_like(b)
    info = P.gpu.solve(b, x, tol=1e-8, restart=30, max_it=300)
    assert info.converged and oi.converged
    assert info.iterations == oi.iterations, (info.iterations, oi.iterations)
    xg = P.to_oracle(x, L)
    assert np.linalg.norm(xg - xo) <= 1e-10 * np.linalg.norm(xo)
    assert info.true_rel_residual <= 1e-8


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p2_n32", "sphere3d_p2_n8", "ellipsoid3d_p3_n12"])
def test_fgmres_fp32_vcycle(name):
    """FP32 V-cycle under FP64 FGMRES reaches the FP64 true residual 1e-8; its solution differs
    from the oracle's FP64 solution by at most the residual bound kappa * 2 tol (Sec. 5)."""
    P = pair(name, "f32")
    F = P.H.finest
    L = len(P.H.levels) - 1
    bo = F.disc.rhs()
    xo, oi = K.fgmres(lambda v: F.A @ v, P.H.vcycle, bo, tol=1e-8, m=30, max_it=300)
    b = P.gpu.rhs()
    x = torch.zeros_like(b)
    info = P.gpu.solve(b, x, tol=1e-8, restart=30, max_it=300)
    assert info.converged and info.true_rel_residual <= 1e-8
    xg = P.to_oracle(x, L)
    # true residual recomputed by the oracle
    assert np.linalg.norm(bo - F.A @ xg) <= 1.01e-8 * np.linalg.norm(bo)
    A = F.A.toarray() if F.N <= 6000 else None
    if A is not None:
        kappa = np.linalg.cond(A)
        assert np.linalg.norm(xg - xo) <= kappa * 2e-8 * np.linalg.norm(xo)
    assert abs(info.iterations - oi.iterations) <= max(2, oi.iterations // 5)


@pytest.mark.parametrize("n,nv", [(1, 1), (1000, 5), (912582, 31), (4097, 32)])
def test_gram_schmidt_dots(n, nv):
    """a6: the FGMRES projections V^T w (deterministic two-stage reduction) against NumPy FP64,
    within the dot-product rounding bound n eps sum_i |V_ki w_i|; bitwise repeatable."""
    P = pair("disk2d_p1_n32")
    rng = np.random.default_rng(n)
    V, w = rng.normal(size=(nv, n)), rng.normal(size=n)
    Vt, wt = torch.tensor(V, device="cuda"), torch.tensor(w, device="cuda")
    out = P.gpu.dots(Vt, wt).cpu().numpy()
    bound = n * 2.2e-16 * (np.abs(V) @ np.abs(w))
    assert np.all(np.abs(out - V @ w) <= bound + 1e-300)
    assert np.array_equal(out, P.gpu.dots(Vt, wt).cpu().numpy())


def test_cluster_tail_is_one_launch():
    """On a hierarchy of small p = 1 levels the whole V-cycle is one cluster launch or one one-CTA
    launch; with the tail disabled it is one launch per phase."""
    import paper_2506_12899_gb300 as S
    P, C, Q = pair("disk2d_p1_n32", tail=16), pair("disk2d_p1_n32", tail=1), pair("disk2d_p1_n32", tail=0)
    r = torch.tensor(W.random_vector(P.H.finest.N, 1), device="cuda")
    for g, expect in ((P.gpu, 1), (C.gpu, 1), (Q.gpu, None)):
        g.vcycle(r)
        torch.cuda.synchronize()
        n0 = S.kernel_launches()
        g.vcycle(r)
        torch.cuda.synchronize()
        n = S.kernel_launches() - n0
        if expect is not None:
            assert n == expect
        else:
            assert n > 10


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p2_n32", "sphere3d_p2_n8", "ellipsoid3d_p3_n12"])
@pytest.mark.parametrize("tail,basis", [(16, 0), (1, 0), (0, 1)], ids=["cluster_tail", "cta_tail", "fp64_basis"])
def test_fgmres_fp64_variants(name, tail, basis):
    """FGMRES with the cluster V-cycle tail, and with the FP64 Krylov basis instead of the
    double-float one: same iteration count and solution (1e-10) as the oracle."""
    P = pair(name, tail=tail, basis=basis)
    F = P.H.finest
    L = len(P.H.levels) - 1
    bo = F.disc.rhs()
    xo, oi = K.fgmres(lambda v: F.A @ v, P.H.vcycle, bo, tol=1e-8, m=30, max_it=300)
    b = P.gpu.rhs()
    x = torch.zeros_like(b)
    info = P.gpu.solve(b, x, tol=1e-8, restart=30, max_it=300)
    assert info.converged and info.iterations == oi.iterations
    assert np.linalg.norm(P.to_oracle(x, L) - xo) <= 1e-10 * np.linalg.norm(xo)


def test_solve_host_buffers():
    P = pair("disk2d_p1_n32")
    b = P.gpu.rhs()
    x = torch.zeros_like(b)
    info_dev = P.gpu.solve(b, x, tol=1e-8)
    bh = b.cpu().numpy().copy()
    xh = np.zeros_like(bh)
    info = P.gpu.solve_host(bh, xh, tol=1e-8)
    assert info.iterations == info_dev.iterations
    assert np.abs(xh - x.cpu().numpy()).max() <= 1e-14 * np.abs(xh).max()


def test_solve_edge_cases():
    import paper_2506_12899_gb300 as S
    P = pair("disk2d_p1_n32")
    b = P.gpu.rhs()
    # b = 0 gives x = 0 without iterating
    z = torch.zeros_like(b)
    x = torch.ones_like(b)
    info = P.gpu.solve(z, x)
    assert info.converged and info.iterations == 0 and float(x.abs().max()) == 0.0
    # iteration cap: SBM_ERR_NOT_CONVERGED, x still improved
    x = torch.zeros_like(b)
    info = P.gpu.solve(b, x, tol=1e-14, max_it=3)
    assert not info.converged and info.status == -4 and info.iterations == 3
    # non-finite right-hand side: SBM_ERR_NAN
    bn = b.clone()
    bn[5] = float("nan")
    with pytest.raises(S.SbmError) as e:
        P.gpu.solve(bn, torch.zeros_like(b))
    assert e.value.code == -5
    # nonzero initial guess equal to the solution converges immediately
    x = torch.zeros_like(b)
    P.gpu.solve(b, x, tol=1e-10)
    info = P.gpu.solve(b, x, tol=1e-8)
    assert info.converged and info.iterations == 0


def test_single_level_and_tiny_mesh():
    """Degenerate hierarchies: one level (the V-cycle is the direct solve) and a 2x2 mesh."""
    import paper_2506_12899_gb300 as S
    prob = W.disk2d_p1(8, 0).replace(coarsest_n=8)
    g = S.Solver(prob)
    assert g.num_levels == 1
    H = MG.Hierarchy(prob)
    m = _dof_map(g, H.finest, 0)
    r = W.random_vector(H.finest.N, 0)
    z = g.vcycle(torch.tensor(r[m], device="cuda")).cpu().numpy()
    zo = np.linalg.solve(H.finest.A.toarray(), r)[m]
    assert np.abs(z - zo).max() <= 1e-11 * np.abs(zo).max()
    prob = W.Problem(dim=2, n=2, p=1, shape=W.disk(2, 0, radius=0.95), coarsest_n=2)
    g = S.Solver(prob)
    assert g.info()["n_active"] == 4 and g.num_levels == 1
    b = g.rhs()
    x = torch.zeros_like(b)
    info = g.solve(b, x, tol=1e-12)
    assert info.converged and info.iterations == 1        # the preconditioner is the exact inverse


def test_full_size_star512_p2_sampled():
    """The star2d p=2 512^2 workload at full size, in the precision and launch configuration the
    benchmark uses: the apply is checked against oracle rows computed cell by cell on 400
    sampled cells (boundary cells included), and the FP32-preconditioned solve reaches the FP64
    true residual 1e-8, with the residual re-evaluated by the oracle on the sampled cells."""
    import paper_2506_12899_gb300 as S
    from oracle.dgsbm import Discretisation
    from oracle.geometry import LevelGeometry
    prob = W.star2d_p2(512, 0)
    g = S.Solver(prob, "f32")
    geom = LevelGeometry(prob, 512, 2)
    D = Discretisation(prob, geom, assemble=False)
    coords = g.layout()
    lin = coords[:, 0].astype(np.int64) + 512 * coords[:, 1].astype(np.int64)
    perm = geom.bg2act[lin]
    assert (perm >= 0).all() and len(perm) == geom.n_active
    inv = np.empty_like(perm)
    inv[perm] = np.arange(len(perm))                 # oracle cell -> compact cell
    nb = D.nb
    rng = np.random.default_rng(0)
    bcells = np.array(sorted({f[0] for f in geom.faces}))
    sample = np.concatenate([rng.choice(geom.n_active, 300, replace=False), rng.choice(bcells, 100, replace=False)])

    def rows(xc):                                    # oracle (A x) on the sampled oracle cells
        X = xc.reshape(-1, nb)
        out = []
        for a in sample:
            y = D.diag_block(a) @ X[inv[a]]
            for nbc, B in D.offdiag_blocks(a):
                y = y + B @ X[inv[nbc]]
            out.append(y)
        return np.array(out)

    x = W.random_vector(g.n_dof(), 3)
    y = g.apply(torch.tensor(x, device="cuda")).cpu().numpy().reshape(-1, nb)[inv[sample]]
    yo = rows(x)
    assert np.abs(y - yo).max() <= 1e-12 * np.abs(yo).max()
    b = g.rhs()
    bo = D.rhs().reshape(-1, nb)
    assert np.abs(b.cpu().numpy().reshape(-1, nb)[inv[sample]] - bo[sample]).max() <= 1e-13 * np.abs(bo).max()
    xs = torch.zeros_like(b)
    info = g.solve(b, xs, tol=1e-8, restart=30, max_it=300)
    assert info.converged and info.true_rel_residual <= 1e-8
    res = bo[sample] - rows(xs.cpu().numpy())
    assert np.abs(res).max() <= 1e-7 * np.abs(bo).max()


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p2_n32", "star2d_p3_n16", "sphere3d_p1_n8", "sphere3d_p2_n8",
                                  "ellipsoid3d_p3_n12"])
def test_staged_kernels(name):
    """The staged thread-per-cell kernels (cells and face neighbours copied into shared memory by
    the CTA before the per-cell arithmetic), forced on every FP32 launch they cover (2D p <= 3,
    3D p <= 2): operator, residual, both sweep directions on every level above the coarsest, and
    the V-cycle, against the oracle with the FP32 bounds used above."""
    import paper_2506_12899_gb300 as S
    P = pair(name)
    g = S.Solver(P.prob, "f32", staged_min_cells=1)
    for l, lev in enumerate(P.H.levels):
        x = W.random_vector(lev.N, 70 + l)
        yo = lev.A @ x
        scale = np.abs(abs(lev.A) @ np.abs(x)).max()
        y32 = P.to_oracle(g.apply(P.to_gpu(x, l, torch.float32), level=l), l)
        assert np.abs(y32 - yo).max() <= 2e-6 * scale, (l, np.abs(y32 - yo).max() / scale)
        f = W.random_vector(lev.N, 80 + l)
        r32 = P.to_oracle(g.residual(P.to_gpu(f, l, torch.float32), P.to_gpu(x, l, torch.float32), level=l), l)
        assert np.abs(r32 - (f - yo)).max() <= 2e-6 * (scale + np.abs(f).max())
        if l == 0:
            continue
        u0 = W.random_vector(lev.N, 90 + l)
        for reverse in (False, True):
            uo = lev.coloured_sweep(u0.copy(), f, reverse=reverse)
            u32 = g.smooth(P.to_gpu(f, l, torch.float32), P.to_gpu(u0, l, torch.float32), level=l, reverse=reverse)
            assert rel_max(P.to_oracle(u32, l), uo) <= 2e-4, (l, reverse, rel_max(P.to_oracle(u32, l), uo))
    L = len(P.H.levels) - 1
    r = W.random_vector(P.H.finest.N, 23)
    zo = P.H.vcycle(r)
    z32 = P.to_oracle(g.vcycle(P.to_gpu(r, L, torch.float32)), L)
    assert np.linalg.norm(z32 - zo) <= 1e-4 * np.linalg.norm(zo), np.linalg.norm(z32 - zo) / np.linalg.norm(zo)
    b = g.rhs()
    xs = torch.zeros_like(b)
    info = g.solve(b, xs, tol=1e-8)
    assert info.converged and info.true_rel_residual <= 1e-8
    g.close()


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "star2d_p3_n16", "sphere3d_p2_n8", "ellipsoid3d_p3_n12",
                                  "complex2d_p1_l3", "complex2d_p2_l2", "complex2d_p3_l2"])
def test_l2_error_matches_oracle(name):
    """sbm_l2_error (Sec. 5.1 / 5.4 error measure) against the oracle's l2_error, on the oracle's own
    direct solution mapped to the library layout and on a random vector."""
    import scipy.sparse.linalg as spla
    P = pair(name)
    F = P.H.finest
    L = len(P.H.levels) - 1
    xo = spla.spsolve(F.A.tocsc(), F.disc.rhs())
    for x in (xo, W.random_vector(F.N, 3)):
        eo = F.disc.l2_error(x)
        eg = P.gpu.l2_error(P.to_gpu(x, L))
        assert abs(eg - eo) <= 1e-10 * eo, (eg, eo)


@pytest.mark.parametrize("p,level,lam", [(1, 3, 1.0), (2, 2, 0.5), (3, 2, 0.75)])
def test_complex2d_solution_and_error(p, level, lam):
    """The complex deformed domain of Sec. 5.4 (Newton closest points on a non-convex level set):
    the GPU FP64 solve reproduces the oracle's direct solution and its L2 error, with the paper's
    tolerance 1e-12."""
    import scipy.sparse.linalg as spla
    import paper_2506_12899_gb300 as S
    prob = W.paper_complex2d(level, p, lam)
    P = Pair(prob)
    F = P.H.finest
    L = len(P.H.levels) - 1
    xo = spla.spsolve(F.A.tocsc(), F.disc.rhs())
    b = P.gpu.rhs()
    x = torch.zeros_like(b)
    info = P.gpu.solve(b, x, tol=1e-12, restart=30, max_it=300)
    assert info.converged
    xg = P.to_oracle(x, L)
    assert np.linalg.norm(xg - xo) <= 1e-9 * np.linalg.norm(xo)
    eo = F.disc.l2_error(xo)
    assert abs(P.gpu.l2_error(x) - eo) <= 1e-6 * eo


@pytest.mark.parametrize("name", ["star2d_p2_n32_redblack", "disk2d_p1_n32_jacobi", "star2d_p3_n16_chebyshev",
                                  "ellipsoid3d_p3_n12_jacobi"])
def test_smoother_variant_launches(name):
    """Launch counts of one V-cycle follow the variant: red-black takes 2 smoother launches per
    sweep instead of d+1; the additive smoothers take no one-launch tail; every variant's FP32
    V-cycle agrees with the oracle's V-cycle within the FP32 bound."""
    import paper_2506_12899_gb300 as S
    P = pair(name)
    L = len(P.H.levels) - 1
    r = W.random_vector(P.H.finest.N, 5)
    g = S.Solver(P.prob, "f32")
    rt = P.to_gpu(r, L, torch.float32)
    g.vcycle(rt)
    torch.cuda.synchronize()
    n0 = S.kernel_launches()
    z = g.vcycle(rt)
    torch.cuda.synchronize()
    n = S.kernel_launches() - n0
    zo = P.H.vcycle(r)
    assert np.linalg.norm(P.to_oracle(z, L) - zo) <= 1e-4 * np.linalg.norm(zo)
    assert n > 2 * (len(P.H.levels) - 1)                 # per-level launches, no one-launch tail
    if P.prob.ordering == 1 and P.prob.smoother == 0:
        u = P.to_gpu(W.random_vector(P.H.finest.N, 6), L, torch.float32)
        f = P.to_gpu(W.random_vector(P.H.finest.N, 7), L, torch.float32)
        n0 = S.kernel_launches()
        g.smooth(f, u)
        assert S.kernel_launches() - n0 == 2
    g.close()


@pytest.mark.parametrize("name,prob", [
    ("star2d_p2_n64", W.star2d_p2(64, 3)),
    ("ellipsoid3d_p3_n24", W.ellipsoid3d_p3(24, 1)),
    ("complex2d_p2_l4", W.paper_complex2d(4, 2, 0.5)),
    ("random_star2d_p3_n32", W.random_star2d_p3(32, 1007)),
    ("sphere3d_p1_n16", W.sphere3d(16, 1, 2)),
])
def test_device_geometry_matches_host(name, prob):
    """The set-up's volume fractions (sub-cell sampling of phi, Sec. 2.1) and closest-point Newton
    solves (Sec. 4.2, Eqs. 19-22) as device kernels: every level's active cells, compact order and
    surrogate faces equal the host set-up's bit for bit, and the shift vectors agree within 1e-12."""
    import paper_2506_12899_gb300 as S
    gd = S.Solver(prob, "f32", device_geometry=1)
    gh = S.Solver(prob, "f32", device_geometry=-1)
    assert gd.num_levels == gh.num_levels
    for l in range(gd.num_levels):
        assert gd.info(l) == gh.info(l)
        assert np.array_equal(gd.layout(l), gh.layout(l))
        cd, sd, dd = gd.export_geometry(l)
        ch, sh, dh = gh.export_geometry(l)
        assert np.array_equal(cd, ch) and np.array_equal(sd, sh)
        assert np.abs(dd - dh).max(initial=0.0) <= 1e-12, (l, np.abs(dd - dh).max())
    gd.close()
    gh.close()


@pytest.mark.parametrize("name,kw,offset", [
    ("disk16", dict(), 0), ("disk16", dict(omega=0.8, ssor_each=1), 0), ("disk16", dict(pre_smooth=0, post_smooth=2), 1),
    ("disk64", dict(coarsest_n=16), 0), ("star64", dict(pre_smooth=2), 0), ("sphere8", dict(), 1),
    ("sphere16", dict(omega=0.9, post_smooth=2), 0), ("sphere32", dict(), 0)])
def test_cta_tail_matches_per_level_launches(name, kw, offset):
    """The one-CTA tail against the per-level launches, both FP32: whole V-cycles inside the tail (vectors at
    an odd offset too), a coarse inverse too large to stage, boundary self blocks in and out of shared
    memory, omega, SSOR and step counts.  Bound: FP32 sums in another order, 2e-5 relative."""
    import paper_2506_12899_gb300 as S
    prob = {"disk16": W.disk2d_p1(16, 1), "disk64": W.disk2d_p1(64, 2), "star64": W.star2d_p2(64, 1).replace(p=1),
            "sphere8": W.sphere3d(8, 1, 1), "sphere16": W.sphere3d(16, 1, 2), "sphere32": W.sphere3d(32, 1, 0)}[name].replace(**kw)
    a, b = S.Solver(prob, "f32"), S.Solver(prob, "f32", tail_max_cells=-1)
    n = a.n_dof()
    r = torch.rand(n + 1, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda")[offset:offset + n] - 0.5
    z = torch.empty(n + 1, device="cuda")[offset:offset + n]
    before = S.kernel_launches()
    a.vcycle(r, z)
    used = S.kernel_launches() - before
    ref = b.vcycle(r.clone())
    assert used < S.kernel_launches() - before - used                 # the tail ran
    assert (z - ref).norm() <= 2e-5 * ref.norm()


@pytest.mark.parametrize("n,p,kw", [(4, 2, dict()), (6, 3, dict()), (8, 2, dict(omega=0.7)), (10, 3, dict(ordering=1)),
                                    (12, 2, dict(ordering=1, omega=0.9)), (14, 2, dict())])
def test_plane_smoother_edges(n, p, kw):
    """The 3D p = 2, 3 smoother (one lane per plane of an interior cell) against the thread-per-DoF kernel, both
    FP32, with last warps of 1 to 10 cells, both orders, relaxation, red-black; and inside a V-cycle, where the
    first sweep reads later colours as zero.  Bound: FP32 sums in another order, 2e-5 relative."""
    import paper_2506_12899_gb300 as S
    prob = W.sphere3d(n, 2, 1).replace(p=p, coarsest_n=4, omega_p3=kw.get("omega", 0.8), **kw)
    a, b = S.Solver(prob, "f32"), S.Solver(prob, "f32", cell_kernel_min_cells=-1, tail_max_cells=-1)
    g = torch.Generator(device="cuda").manual_seed(n)
    f, u = (torch.rand(a.n_dof(), generator=g, device="cuda") - 0.5 for _ in range(2))
    for rev in (False, True):
        x, y = a.smooth(f, u.clone(), reverse=rev), b.smooth(f, u.clone(), reverse=rev)
        assert (x - y).norm() <= 2e-5 * y.norm()
    z, ref = a.vcycle(f), b.vcycle(f)
    assert (z - ref).norm() <= 2e-5 * ref.norm()


def _crc(t):
    return zlib.crc32(t.cpu().numpy().tobytes())


def _f32(rng, n):
    return torch.from_numpy(rng.uniform(-1, 1, n).astype(np.float32)).cuda()


@pytest.mark.parametrize("n,p,omega,forward,reverse", [
    (12, 2, 1.0, 0x4098c97d, 0x9ee396b1), (14, 2, 0.7, 0x272a8730, 0xe95451d6),
    (10, 3, 0.8, 0xbd815a6d, 0xaa72d618), (12, 3, 1.0, 0xc6263fa2, 0x9ef98190)])
def test_plane_smoother_keeps_the_bits_of_the_line_form(n, p, omega, forward, reverse):
    """The 3D p = 2, 3 FP32 sweep adds its terms in the order of the kernel with one lane per x-line that it
    replaced, to the same bits: CRC-32 of the results, taken with that kernel (commit e2b57b5).  The number of
    steps of long 3D solves depends on these bits."""
    import paper_2506_12899_gb300 as S
    a = S.Solver(W.sphere3d(n, 2, 1).replace(p=p, coarsest_n=4, omega=omega, omega_p3=omega), "f32")
    rng = np.random.default_rng(n)
    f, u = _f32(rng, a.n_dof()), _f32(rng, a.n_dof())
    assert _crc(a.smooth(f, u.clone())) == forward
    assert _crc(a.smooth(f, u.clone(), reverse=True)) == reverse


@pytest.mark.parametrize("n,geometry,kw,crc", [
    (8, 1, dict(), 0x24558b36), (16, 2, dict(), 0xc9b6694c), (16, 0, dict(omega=0.9, post_smooth=2), 0x596c327b),
    (16, 3, dict(ssor_each=1), 0xd8f94f8d), (32, 1, dict(pre_smooth=0, post_smooth=2), 0x475e82af),
    (32, 0, dict(), 0xed805dea)])
def test_3d_tail_keeps_its_bits(n, geometry, kw, crc):
    """V-cycles of 3D p = 1 spheres, inside the one-CTA tail (8^3, 16^3) and above it, to the bits of the tail's
    first form (CRC-32 of the results, commit e2b57b5), for the same reason."""
    import paper_2506_12899_gb300 as S
    a = S.Solver(W.sphere3d(n, 1, geometry).replace(**kw), "f32")
    assert _crc(a.vcycle(_f32(np.random.default_rng(n), a.n_dof()))) == crc


@pytest.mark.parametrize("name", ["sphere3d_p3", "star2d_p2", "sphere3d_p1"])
def test_vcycle_blocks_are_held_for_the_precisions_used(name):
    """FP64 self blocks of the levels below the finest belong to the FP64 V-cycle: an FP32 solver holds them only
    from its first FP64 V-cycle on.  Either solver runs V-cycles of either precision to the same bits."""
    import paper_2506_12899_gb300 as S
    prob = {"sphere3d_p3": W.sphere3d(40, 2, 0).replace(p=3, coarsest_n=4), "star2d_p2": W.star2d_p2(64, 0),
            "sphere3d_p1": W.sphere3d(16, 1, 0)}[name]

    def held(precision):                               # bytes of device memory a set-up takes
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        s = S.Solver(prob, precision)
        return s, free - torch.cuda.mem_get_info()[0]

    for precision in ("f32", "f64"):                   # code is loaded
        held(precision)[0].close()
    a, small = held("f32")
    b, large = held("f64")
    blocks = 0
    for l in range(a.num_levels - 1):
        info = a.info(l)
        blocks += info["n_boundary"] * (info["n_dof"] // info["n_active"]) ** 2 * 8
    assert small <= large - blocks + (4 << 20), (small, large, blocks)   # allocations come in 2 MB pieces
    r = _f32(np.random.default_rng(1), a.n_dof())
    for x in (r, r.double()):
        assert torch.equal(a.vcycle(x), b.vcycle(x))
