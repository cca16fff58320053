"""Waits of the team solver that run out: with a limit of one clock cycle (MPCG_TIMEOUT_CYCLES) a solve
whose CTAs wait long for one another ends in MPCG_ERR_TIMEOUT, and the context goes on to solve the same
system with the usual limit. The whole grid waits for the CTA that holds a row of a million nonzeros
(every CTA of the others polls some 30 us before it looks at the limit, the row takes longer); a
cluster waits for the CTA that runs 40,000 levels of an IC(0) application, and its ring of level blocks
is in use then."""
import numpy as np
import pytest

from paper_2504_14268_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TIMEOUT = 5  # MPCG_ERR_TIMEOUT


@pytest.fixture(scope="module")
def M():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2504_14268_gb300 import mpcg

    return mpcg


def _arrow(n):
    """Diagonal 4, and entries 1 / n in the first row and column."""
    i = np.arange(1, n)
    rp = np.concatenate([[0], n + 2 * np.arange(n)])
    ci, val = np.empty(rp[-1], dtype=np.int32), np.empty(rp[-1])
    ci[:n], val[:n] = np.arange(n), 1.0 / n
    val[0] = 4.0
    ci[n::2], val[n::2] = 0, 1.0 / n
    ci[n + 1::2], val[n + 1::2] = i, 4.0
    return n, rp.astype(np.int32), ci, val


def _tridiagonal(n):
    i = np.arange(n)
    r = np.concatenate([i, i[1:], i[:-1]])
    c = np.concatenate([i, i[:-1], i[1:]])
    v = np.concatenate([np.full(n, 4.0), np.full(2 * n - 2, -1.0)])
    o = np.lexsort((c, r))
    return n, np.concatenate([[0], np.cumsum(np.bincount(r))]).astype(np.int32), c[o].astype(np.int32), v[o]


@pytest.mark.parametrize("A,precond", [(_arrow(1_000_000), 0), (_tridiagonal(20_000), 2)], ids=["grid", "cluster_ic0"])
def test_a_wait_that_runs_out_is_an_error(M, monkeypatch, A, precond):
    n, rp, ci, val = A
    ctx = M.Context(0, M.Options(min_k=0, precond=precond))
    mat = ctx.matrix((n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda()))
    if precond == 2:
        mat.ic0()
    b = torch.as_tensor(np.random.default_rng(1).uniform(-1, 1, n)).cuda()
    x = torch.zeros_like(b)
    pol = ctx.policy_fixed((4, 4, 4, 4))
    want, _ = ctx.solve(mat, b, x, 1e-8, 30, pol)
    ref = x.clone()
    for _ in range(3):
        monkeypatch.setenv("MPCG_TIMEOUT_CYCLES", "1")
        with pytest.raises(M.MpcgError) as e:
            ctx.solve(mat, b, x, 1e-8, 30, pol)
        assert e.value.status == TIMEOUT
        monkeypatch.delenv("MPCG_TIMEOUT_CYCLES")
        res, _ = ctx.solve(mat, b, x, 1e-8, 30, pol)
        assert (res["outcome"], res["iters"]) == (want["outcome"], want["iters"])
        assert torch.equal(x, ref)
