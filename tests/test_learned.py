"""Learned boundary-cell correction on the GPU against the FP64 oracle (oracle/learned.py).

The library computes features and the correction in BF16 with FP32 accumulation, so parity
bounds come from the BF16 unit roundoff (2^-9 relative per rounding):
  * features: each value is one BF16 rounding of an FP64 quantity: |x - x_o| <= 2^-8 |x_o|;
    the norms s (FP32 sums of squares) to 1e-5 relative;
  * MLP forward: inputs, weights and both hidden activations rounded to BF16, FP32 sums:
    relative L2 error of the outputs <= 1e-2;
  * gradients (BF16 dY, dZ and activations): cosine >= 0.999, relative L2 error <= 2e-2;
  * V-cycle with the correction: the correction part (z_learned - z_plain) to 2e-2 relative L2,
    the plain part to the FP64 V-cycle bound.
"""
import os
import tempfile

import numpy as np
import pytest

import workloads as W
from oracle import learned as OL

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from _pairs import Pair  # noqa: E402

_cache = {}


def pair(name):
    if name not in _cache:
        prob = {"star2d_p2_n32": W.star2d_p2(32, 1), "disk2d_p1_n32": W.disk2d_p1(32, 0),
                "sphere3d_p1_n8": W.sphere3d(8, 1, 2), "star2d_p3_n16": W.star2d_p2(16, 2).replace(p=3)}[name]
        _cache[name] = Pair(prob)
    return _cache[name]


def bnd_cells_oracle(P):
    """Oracle active indices of the library's boundary cells, in the library's order."""
    F = P.H.finest
    nb = F.nb
    cells = P.gpu.learned_cells()
    m = P.maps[-1].reshape(-1, nb)[:, 0] // nb          # compact cell -> oracle active index
    return m[cells]


def mlp_pair(P, hidden=32, seed=3):
    import paper_2506_12899_gb300 as S
    lev = P.H.finest
    F = OL.feature_size(P.prob.dim, lev.p)
    net = OL.MLP(F, hidden, lev.nb, seed=seed)
    gm = S.Mlp(P.prob.dim, lev.p, hidden)
    assert (gm.F, gm.O) == (F, lev.nb)
    gm.set_params(net.params())
    # the oracle runs with the FP32-rounded parameters the library stores
    for a in net.params():
        a[...] = a.astype(np.float32).astype(np.float64)
    return net, gm


@pytest.mark.parametrize("name", ["star2d_p2_n32", "sphere3d_p1_n8", "star2d_p3_n16"])
def test_features_match_oracle(name):
    """Features and patch norms of every boundary cell from a random residual."""
    P = pair(name)
    lev = P.H.finest
    r = W.random_vector(lev.N, 5)
    X, s = P.gpu.learned_features(P.to_gpu(r, len(P.H.levels) - 1), OL.feature_size(P.prob.dim, lev.p))
    cells = bnd_cells_oracle(P)
    assert sorted(cells.tolist()) == sorted(int(c) for c in OL.boundary_cells(lev))
    Xo, so = OL.features(lev, r, cells)
    Xg = X.double().cpu().numpy()
    assert np.all(np.abs(Xg - Xo) <= 2.0 ** -8 * np.abs(Xo) + 1e-30), np.abs(Xg - Xo).max()
    assert np.allclose(s.double().cpu().numpy(), so, rtol=1e-5, atol=0)


def test_forward_matches_oracle():
    P = pair("star2d_p2_n32")
    net, gm = mlp_pair(P)
    rng = np.random.default_rng(0)
    X = rng.uniform(-1, 1, size=(300, gm.F))
    Y = gm.forward(torch.tensor(X, dtype=torch.float32, device="cuda")).double().cpu().numpy()
    Yo = net.forward(X)
    assert np.linalg.norm(Y - Yo) <= 1e-2 * np.linalg.norm(Yo)


def test_gradients_match_oracle():
    P = pair("star2d_p2_n32")
    net, gm = mlp_pair(P)
    rng = np.random.default_rng(1)
    X = rng.uniform(-1, 1, size=(257, gm.F))
    T = rng.normal(size=(257, gm.O))
    loss, g = gm.gradients(torch.tensor(X, dtype=torch.float32, device="cuda"),
                           torch.tensor(T, dtype=torch.float32, device="cuda"))
    Yo = net.forward(X)
    go = np.concatenate([a.reshape(-1) for a in net.backward(Yo, T)])
    assert abs(loss - net.loss(Yo, T)) <= 1e-2 * net.loss(Yo, T)
    cos = g @ go / (np.linalg.norm(g) * np.linalg.norm(go))
    assert cos >= 0.999, cos
    assert np.linalg.norm(g - go) <= 2e-2 * np.linalg.norm(go)


@pytest.mark.parametrize("name", ["star2d_p2_n32", "sphere3d_p1_n8"])
def test_vcycle_with_correction_matches_oracle(name):
    """z = V(r) with the correction after the finest post-smoothing (in units of s h^(2-d)), against
    the oracle hook."""
    P = pair(name)
    net, gm = mlp_pair(P, seed=7)
    for a in (net.W3, net.b3):                           # keep the correction a modest fraction of z
        a *= 0.05
    gm.set_params(net.params())
    L = len(P.H.levels) - 1
    r = W.random_vector(P.H.finest.N, 9)
    P.gpu.attach_mlp(None)
    z_plain = P.to_oracle(P.gpu.vcycle(P.to_gpu(r, L)), L)
    P.gpu.attach_mlp(gm, scale=1.0)
    try:
        z_learn = P.to_oracle(P.gpu.vcycle(P.to_gpu(r, L)), L)
    finally:
        P.gpu.attach_mlp(None)
    zo_plain = P.H.vcycle(r.copy())
    zo_learn = P.H.vcycle(r.copy(), correction=OL.correction(net, bnd_cells_oracle(P)))
    assert np.abs(z_plain - zo_plain).max() <= 1e-10 * np.abs(zo_plain).max()
    d, do = z_learn - z_plain, zo_learn - zo_plain
    assert np.linalg.norm(do) > 1e-6 * np.linalg.norm(zo_plain)
    assert np.linalg.norm(d - do) <= 2e-2 * np.linalg.norm(do)


@pytest.mark.parametrize("name", ["disk2d_p1_n32", "sphere3d_p1_n8"])
def test_collect_matches_oracle_targets(name):
    """Collected pairs: features of r = -A u and targets -u_K / (s_K h^(2-d)) after one plain V-cycle
    step; then the targets normalised to unit RMS (sbm_mlp_target_scale)."""
    import paper_2506_12899_gb300 as S
    P = pair(name)
    lev = P.H.finest
    L = len(P.H.levels) - 1
    gm = S.Mlp(P.prob.dim, lev.p, 16)
    u0 = W.random_vector(lev.N, 21)
    n = P.gpu.collect(gm, P.to_gpu(u0, L)[None, :].contiguous(), 1)
    cells = bnd_cells_oracle(P)
    assert n == len(cells) and gm.num_samples() == n
    # oracle: one step of u <- u + V(-A u) from the same start, the pair of each boundary cell in
    # the library's cell order
    Xo, To = OL.training_pairs(P.H, 1, 1, 0, u0s=[u0], cells=cells)
    assert Xo.shape[0] == n
    # the library keeps the pairs internally; train for zero epochs is a no-op, so read them back
    # through the loss of an MLP whose output is exactly zero: loss = mean(T^2)
    zero = [np.zeros_like(a) for a in OL.MLP(gm.F, gm.H, gm.O).params()]
    gm.set_params(zero)
    loss = gm.train(epochs=1, batch=n, lr=1e-12)
    assert abs(loss - np.mean(To ** 2)) <= 1e-4 * np.mean(To ** 2)
    rms = gm.target_scale()
    assert abs(rms - np.sqrt(np.mean(To ** 2))) <= 1e-5 * rms
    gm.set_params(zero)
    loss = gm.train(epochs=1, batch=n, lr=1e-12)
    assert abs(loss - 1.0) <= 1e-4


def test_training_reduces_loss():
    import paper_2506_12899_gb300 as S
    P = pair("disk2d_p1_n32")
    gm = S.Mlp(2, 1, 32, seed=1)
    g = torch.Generator(device="cuda").manual_seed(0)
    u0 = (2 * torch.rand((4, P.gpu.n_dof()), generator=g, device="cuda", dtype=torch.float64) - 1).contiguous()
    P.gpu.collect(gm, u0, 3)
    first = gm.train(epochs=1, batch=64, lr=1e-3, seed=0)
    last = gm.train(epochs=30, batch=64, lr=1e-3, seed=1)
    assert np.isfinite(first) and last < 0.8 * first, (first, last)


def test_fallback_switches_off_a_bad_correction():
    """An MLP far worse than plain (large random output layer) must trigger the fallback; the
    solve then converges with the plain V-cycle (FGMRES tolerates the preconditioner change)."""
    import paper_2506_12899_gb300 as S
    P = pair("star2d_p2_n32")
    b = P.gpu.rhs()
    x = torch.zeros_like(b)
    plain = P.gpu.solve(b, x)
    rate = plain.true_rel_residual ** (1.0 / plain.iterations)
    net, gm = mlp_pair(P, seed=11)
    net.W3 *= 1e3
    gm.set_params(net.params())
    P.gpu.attach_mlp(gm, scale=1.0, fallback_rate=rate)
    try:
        x.zero_()
        info = P.gpu.solve(b, x)
    finally:
        P.gpu.attach_mlp(None)
    assert info.learned and info.learned_fallback and info.converged
    assert info.true_rel_residual <= 1e-8
    # without the rule the same MLP is used throughout: still a valid flexible preconditioner or not,
    # but the flags must say so
    P.gpu.attach_mlp(gm, scale=1.0, fallback_rate=0.0)
    try:
        x.zero_()
        info2 = P.gpu.solve(b, x, max_it=5)
    finally:
        P.gpu.attach_mlp(None)
    assert info2.learned and not info2.learned_fallback


def test_checkpoint_roundtrip_and_corruption():
    import paper_2506_12899_gb300 as S
    gm = S.Mlp(2, 2, 24, seed=5)
    w = gm.get_params()
    with tempfile.TemporaryDirectory() as d:
        path = os.path.join(d, "m.bin")
        gm.save(path)
        other = S.Mlp(2, 2, 24, seed=6)
        assert not np.array_equal(other.get_params(), w)
        other.load(path)
        assert np.array_equal(other.get_params(), w)
        raw = bytearray(open(path, "rb").read())
        raw[100] ^= 0x40                                  # one flipped bit in the weights
        open(path, "wb").write(bytes(raw))
        with pytest.raises(S.SbmError):
            other.load(path)
        wrong = S.Mlp(2, 2, 16)
        gm.save(path)
        with pytest.raises(S.SbmError):
            wrong.load(path)


@pytest.mark.parametrize("dim,p,hidden,rows", [(2, 2, 128, 1000), (2, 1, 32, 77), (3, 1, 128, 300), (2, 3, 64, 4096)])
def test_tensor_core_gemm_matches_mma_sync(dim, p, hidden, rows):
    """The tcgen05 tensor-core GEMMs (default) and the warp-level mma.sync GEMMs compute the same
    BF16 products with FP32 sums: forward outputs and gradients agree within the FP32 summation
    differences (1e-4 relative), on ragged shapes (rows, F, O not multiples of the tiles)."""
    import paper_2506_12899_gb300 as S
    gm = S.Mlp(dim, p, hidden, seed=11)
    rng = np.random.default_rng(rows)
    X = torch.tensor(rng.uniform(-1, 1, size=(rows, gm.F)), dtype=torch.float32, device="cuda")
    T = torch.tensor(rng.normal(size=(rows, gm.O)), dtype=torch.float32, device="cuda")
    gm.gemm_backend(0)
    y_tc = gm.forward(X).cpu().numpy()
    l_tc, g_tc = gm.gradients(X, T)
    gm.gemm_backend(1)
    y_ws = gm.forward(X).cpu().numpy()
    l_ws, g_ws = gm.gradients(X, T)
    assert np.linalg.norm(y_tc - y_ws) <= 1e-4 * np.linalg.norm(y_ws)
    assert abs(l_tc - l_ws) <= 1e-4 * l_ws
    assert np.linalg.norm(g_tc - g_ws) <= 1e-3 * np.linalg.norm(g_ws)


@pytest.mark.parametrize("dim,p,hidden,rows", [(2, 1, 8, 1), (2, 2, 33, 127), (3, 1, 128, 128), (2, 3, 200, 129),
                                               (3, 2, 256, 300), (2, 1, 264, 140), (2, 1, 32, 152 * 128 + 5)])
def test_forward_edges_match_mma_sync(dim, p, hidden, rows):
    """The one-launch forward pass (hidden widths up to 256) and the layer-by-layer one (264) against the
    mma.sync layers at the edges of the 128-row tiles, of the padded widths, and past one tile per SM.
    Same BF16 products, FP32 sums in another order: an activation next to a rounding boundary may round
    the other way, one BF16 unit (2^-8) of one hidden value."""
    import paper_2506_12899_gb300 as S
    gm = S.Mlp(dim, p, hidden, seed=3)
    X = torch.rand((rows, gm.F), generator=torch.Generator(device="cuda").manual_seed(rows), device="cuda") * 2 - 1
    y = gm.forward(X)
    gm.gemm_backend(1)
    ref = gm.forward(X)
    assert torch.isfinite(y).all() and (y - ref).norm() <= 2.0 ** -8 * ref.norm()


@pytest.mark.parametrize("dim,p,hidden,rows", [(2, 1, 8, 1), (2, 2, 33, 127), (3, 1, 200, 129), (3, 2, 256, 300),
                                               (2, 1, 264, 140), (2, 3, 128, 1111), (2, 1, 32, 152 * 128 + 5)])
def test_training_pass_edges_match_mma_sync(dim, p, hidden, rows):
    """The one-launch training pass with split weight gradients against the mma.sync layers, as above; the
    gradients round twice (activations, backward products), each at most one BF16 unit of one value."""
    import paper_2506_12899_gb300 as S
    gm = S.Mlp(dim, p, hidden, seed=5)
    g = torch.Generator(device="cuda").manual_seed(rows)
    X = torch.rand((rows, gm.F), generator=g, device="cuda") * 2 - 1
    T = torch.randn((rows, gm.O), generator=g, device="cuda")
    loss, grad = gm.gradients(X, T)
    again, grad2 = gm.gradients(X, T)
    assert loss == again and np.array_equal(grad, grad2)              # fixed-order sums
    gm.gemm_backend(1)
    ref_loss, ref = gm.gradients(X, T)
    assert abs(loss - ref_loss) <= 2.0 ** -8 * ref_loss
    assert np.linalg.norm(grad - ref) <= 2.0 ** -7 * np.linalg.norm(ref)


def test_network_calls_overlap_whatever_solver_was_used_last():
    """The launch mode of a network's calls is its own: an FP64 solver (no overlap by default) used before
    on the same thread does not change it, and a call with a solver and a network follows the solver."""
    import paper_2506_12899_gb300 as S
    prob = W.disk2d_p1(16, 0)
    f64, f32 = S.Solver(prob, "f64"), S.Solver(prob, "f32")
    m = S.Mlp(2, 1, 16)
    X, T = torch.zeros((3, m.F), device="cuda"), torch.zeros((3, m.O), device="cuda")
    for solver, mode in ((f64, False), (f32, True)):
        solver.rhs()
        assert S.launch_overlap() == mode
        m.forward(X)
        assert S.launch_overlap()
        solver.rhs()
        m.gradients(X, T)
        assert S.launch_overlap()
        solver.attach_mlp(m)
        assert S.launch_overlap() == mode


def test_network_stays_usable_after_a_batch_that_does_not_fit():
    """A batch whose buffers cannot be allocated (8 TB) is refused with SBM_ERR_ALLOC before any launch; the
    network then computes smaller batches in buffers of their own, with the same results as before."""
    import ctypes
    import paper_2506_12899_gb300 as S
    m = S.Mlp(3, 3, 264, seed=1)                       # wider than the one-launch kernel: uses the batch buffers
    g = torch.Generator(device="cuda").manual_seed(0)
    X = torch.rand((130, m.F), generator=g, device="cuda") - 0.5
    T = torch.rand((130, m.O), generator=g, device="cuda")
    y, (loss, grad) = m.forward(X), m.gradients(X, T)
    code = S.load_library().sbm_mlp_forward(m.h, ctypes.c_void_p(X.data_ptr()), 2_000_000_000,
                                            ctypes.c_void_p(y.clone().data_ptr()))
    assert S.ERRORS[code] == "SBM_ERR_ALLOC"
    assert torch.equal(m.forward(X[:100].contiguous()), y[:100])
    again = m.gradients(X, T)
    assert again[0] == loss and np.array_equal(again[1], grad)


_ROWS_CASES = [("star", 64, False), ("star", 200, False), ("star", 256, False), ("sphere", 32, True), ("sphere", 200, True)]


def _rows_problem(name):
    return W.random_star2d_p3(64, 1002) if name == "star" else W.sphere3d(128, 1, 0)


@pytest.mark.parametrize("name,hidden,two_tiles", _ROWS_CASES)
def test_attached_correction_matches_mma_sync(name, hidden, two_tiles):
    """The one-launch pass over BF16 feature rows, as an attached V-cycle runs it, against the mma.sync layers:
    widths below and above 128, and more rows than one 128-row tile per SM.  Same BF16 products, FP32 sums in
    another order, so one BF16 unit (2^-8) of one hidden value."""
    import paper_2506_12899_gb300 as S
    a = S.Solver(_rows_problem(name), "f32")
    assert (len(a.learned_cells()) > 152 * 128) == two_tiles
    r = torch.rand(a.n_dof(), generator=torch.Generator(device="cuda").manual_seed(hidden), device="cuda") - 0.5
    plain = a.vcycle(r)
    m = S.Mlp(a.prob.dim, a.prob.p, hidden, seed=7)
    a.attach_mlp(m, scale=1.0)
    z = a.vcycle(r) - plain
    m.gemm_backend(1)
    ref = a.vcycle(r) - plain
    assert ref.norm() > 0 and (z - ref).norm() <= 2.0 ** -8 * ref.norm()


@pytest.mark.parametrize("name,hidden,two_tiles", _ROWS_CASES)
def test_training_on_stored_rows_matches_mma_sync(name, hidden, two_tiles):
    """One training step over the whole stored set (BF16 rows) against the mma.sync layers.  The loss of the
    step differs by BF16 rounding (2^-8).  Adam's first step is lr times the gradient's sign: an entry whose
    gradient is below its rounding error (2^-7 of the gradients' size, as in the pass with FP32 rows) may
    change sign; at most 5% of them are that small, so the steps' cosine is at least 0.9."""
    import paper_2506_12899_gb300 as S
    a = S.Solver(_rows_problem(name), "f32")
    u0 = torch.rand((1, a.n_dof()), generator=torch.Generator(device="cuda").manual_seed(hidden), device="cuda") - 0.5
    step, loss = [], []
    for backend in (0, 1):
        m = S.Mlp(a.prob.dim, a.prob.p, hidden, seed=7)
        rows = a.collect(m, u0, 1)
        assert (rows > 152 * 128) == two_tiles
        m.gemm_backend(backend)
        before = m.get_params()
        loss.append(m.train(epochs=1, batch=rows, lr=1e-3, seed=0))
        step.append((m.get_params() - before).astype(np.float64))
    assert abs(loss[0] - loss[1]) <= 2.0 ** -8 * loss[1]
    cosine = step[0] @ step[1] / (np.linalg.norm(step[0]) * np.linalg.norm(step[1]))
    assert cosine >= 0.9, cosine
