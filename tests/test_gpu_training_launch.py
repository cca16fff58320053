"""Training and collection keep the launch forms whose sums give a seed the same table: rounds of
several systems the lockstep kernel's, one system the persistent kernel's. Tables, counts and
transitions are compared bit for bit with those forms asked for by name."""
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


def _systems(ctx, edges):
    mats, bs = [], []
    for i, m in enumerate(edges):
        A = I.fem27_aniso(m, 1e-2)
        _, b = I.rhs_from_xstar(A, np.random.default_rng(i))
        n, rp, ci, val = A
        mats.append(ctx.matrix((n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda())))
        bs.append(torch.as_tensor(b).cuda())
    return mats, bs


def _train(M, edges, **opts):
    ctx = M.Context(0, M.Options(seed=4, **opts))
    mats, bs = _systems(ctx, edges)
    pol = ctx.policy_qtable(np.zeros((4, 100, 5)), np.zeros((4, 100), dtype=np.int32))
    its = ctx.train_qtable(mats, bs, 1e-8, 24, 3, pol, want_iters=True)
    data = ctx.collect(mats, bs, 1e-8, 24, pol, 0.3, 7)
    return (*pol.qtable(), its, data)


def test_rounds_of_several_systems_are_the_lockstep_kernels(M):
    for a, b in zip(_train(M, [7, 10, 13, 16]), _train(M, [7, 10, 13, 16], batch_mode=2)):
        assert np.array_equal(a, b)


def test_one_system_is_the_persistent_kernels(M, monkeypatch):
    a = _train(M, [9])[:3]  # one CTA: 18,541 units of work
    monkeypatch.setenv("MPCG_FORCE_TEAM", "1")
    for u, v in zip(a, _train(M, [9])[:3]):
        assert np.array_equal(u, v)
