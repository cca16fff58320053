"""Policy states at the ends of the number range: a residual that is not a number lies above every
bin threshold, and decisions near thresholds far below fp32's range are counted like the others."""
import numpy as np
import pytest

from paper_2504_14268_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2504_14268_gb300 import mpcg

    return mpcg


def _dev(A):
    n, rp, ci, val = A
    return (n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda())


def _table():
    """tf32 in the first residual bin, fp64 in the others."""
    Q = np.zeros((4, 100, 5))
    for s in range(100):
        Q[:, s, 2 if s % 10 == 0 else 4] = 1.0
    return Q


@pytest.mark.parametrize("mode", [0, 2])
def test_a_residual_that_is_no_number_is_in_the_first_bin(M, mode):
    ctx = M.Context(0, M.Options(min_k=0, batch_mode=mode))
    mat = ctx.matrix(_dev(I.poisson2d(9)))
    b = torch.ones(81, dtype=torch.float64, device="cuda")
    b[3] = float("inf")  # rho_0 = inf / inf
    x = torch.zeros_like(b)
    res = ctx.solve_batched([mat], [b], [x], [1e-8], [5], ctx.policy_qtable(_table()))[0]
    assert res["outcome"] == 2 and res["iters"] == 0
    assert np.array_equal(res["action_hist"], np.eye(8, dtype=int)[[2, 2, 2, 2]])


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("edge_tol", [0.09, 0.5])
def test_near_edge_count_at_tiny_thresholds(M, mode, edge_tol):
    """Thresholds 10^(-1.875 m) down to 7e-59: the count is that of the recorded residuals."""
    opt = dict(min_k=0, batch_mode=mode, r_bins=32, eps_min=1e-60, edge_tol=edge_tol)
    A = I.poisson2d(12)
    _, b = I.rhs_from_xstar(A, np.random.default_rng(0))
    ctx = M.Context(0, M.Options(**opt))
    mat = ctx.matrix(_dev(A))
    bd = torch.as_tensor(b).cuda()
    pol = ctx.policy_qtable(np.tile([0.0, 0, 0, 0, 1.0], (4, 320, 1)))
    res, hist = ctx.solve(mat, bd, torch.zeros_like(bd), 0.0, 260, pol, history_cap=260)
    rho = np.concatenate([[1.0], hist["rho"][: res["iters"] - 1]])  # of each decision
    assert rho.min() < 1e-50
    thr = 10.0 ** (-1.875 * np.arange(1, 32))
    near = np.abs(rho[:, None] / thr - 1) <= edge_tol
    assert near[:, 20:].any()
    assert res["near_edge_count"] == near.any(1).sum()
    res2, _ = ctx.solve(mat, bd, torch.zeros_like(bd), 0.0, 260, pol)
    assert res2["near_edge_count"] == res["near_edge_count"]
