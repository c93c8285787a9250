"""Failure paths of the bounded waits, on the GPU without a fault: a wait that runs out returns an
error status the host reads, and the device context stays usable.

The staged kernels (Gram-Schmidt sweeps, the V-cycle tail) wait on mbarriers for bulk
asynchronous copies.  sbm_async_wait_selftest runs one such wait with a copy that is announced but
never issued (a phase that nothing completes): the wait gives up after a bounded number of polls,
sets the library's fault flag, and the call returns SBM_ERR_CUDA.  A solve afterwards must still
converge and report no fault.
"""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_bounded_wait_succeeds_when_the_copy_arrives():
    import paper_2506_12899_gb300 as S
    S.async_wait_selftest(False)


def test_bounded_wait_runs_out_and_reports():
    import paper_2506_12899_gb300 as S
    with pytest.raises(S.SbmError) as ei:
        S.async_wait_selftest(True)
    assert "mbarrier wait gave up" in str(ei.value)
    # the flag was cleared by the failing call: the next good wait and a full solve are clean
    S.async_wait_selftest(False)
    g = S.Solver(W.disk2d_p1(16, 0), "f32")
    b = g.rhs()
    x = torch.zeros_like(b)
    info = g.solve(b, x)
    assert info.converged and info.true_rel_residual <= 1e-8


@pytest.mark.parametrize("hidden,rows", [(32, 5), (128, 300), (200, 129)])
def test_network_wait_that_runs_out_is_reported_once(hidden, rows):
    """A wait limit of zero polls: every role of the one-launch kernel gives up at its first wait, the
    outputs are zero, the next synchronising call raises, and the network works again afterwards."""
    import paper_2506_12899_gb300 as S
    m, other = S.Mlp(2, 2, hidden, seed=1), S.Mlp(2, 2, hidden, seed=1)
    X = torch.rand((rows, m.F), device="cuda") - 0.5
    T = torch.zeros((rows, m.O), device="cuda")
    good, (loss, grad) = m.forward(X), m.gradients(X, T)
    assert good.abs().max() > 0
    m.wait_limit(0)
    y = m.forward(X)
    assert torch.equal(y, torch.zeros_like(y))
    other.gradients(X, T)                                # another network is not blamed
    with pytest.raises(S.SbmError, match="in time"):
        m.gradients(X, T)
    m.wait_limit()
    assert torch.equal(m.forward(X), good)
    again = m.gradients(X, T)
    assert again[0] == loss and (again[1] == grad).all()


def test_solve_reports_a_lost_wait_of_its_network():
    """sbm_vcycle with a network whose waits run out applies a zero correction; sbm_solve with it attached
    returns SBM_ERR_CUDA instead of a silent result, and a solver without the network is not affected."""
    import paper_2506_12899_gb300 as S
    prob = W.random_star2d_p3(32, 1001)
    a, plain = S.Solver(prob, "f32"), S.Solver(prob, "f32")
    m = S.Mlp(2, 3, 64, seed=2)
    r = torch.rand(a.n_dof(), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda") - 0.5
    z0 = plain.vcycle(r)
    a.attach_mlp(m, scale=0.01)
    good = a.vcycle(r)
    assert not torch.equal(good, z0)
    m.wait_limit(0)
    assert torch.equal(a.vcycle(r), z0)
    b = a.rhs()
    assert plain.solve(b, torch.zeros_like(b)).converged
    with pytest.raises(S.SbmError, match="learned correction"):
        a.solve(b, torch.zeros_like(b), max_it=2)
    m.wait_limit()
    a.attach_mlp(m, scale=0.01)
    assert torch.equal(a.vcycle(r), good)
    assert a.solve(b, torch.zeros_like(b)).converged
