"""The choice of a launch form does not cost a multiple of what another form takes: a few large systems
as teams against the lockstep kernel, and a single system beyond the whole-grid team's range against the
stepped kernels. Medians of five calls of some milliseconds each; where the choice was wrong they were
1.7 (single system) and 4 times (batch) as long."""
import time

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


def _median(f):
    f()
    t = []
    for _ in range(5):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return sorted(t)[2]


def test_two_large_systems_as_teams(M):
    A = I.fem27_aniso(64, 1e-2)
    b = torch.as_tensor(np.random.default_rng(0).uniform(-1, 1, A[0])).cuda()
    took = []
    for mode in (1, 2):
        ctx = M.Context(0, M.Options(min_k=0, batch_mode=mode))
        mats, bs, xs = [ctx.matrix(_dev(A)) for _ in range(2)], [b, b], [torch.zeros_like(b) for _ in range(2)]
        pol = ctx.policy_fixed((4, 4, 4, 4))
        took.append(_median(lambda: ctx.solve_batched(mats, bs, xs, [0.0] * 2, [30] * 2, pol)))
    assert took[0] < 2 * took[1]


def test_a_system_beyond_the_whole_grid_team(M):
    A = I.poisson2d(1800)  # 3.24e6 rows, just below 2^24 nonzeros
    b = torch.as_tensor(np.random.default_rng(0).uniform(-1, 1, A[0])).cuda()
    took = []
    for stepped in (0, 2):
        ctx = M.Context(0, M.Options(min_k=0, stepped=stepped))
        mat, x, pol = ctx.matrix(_dev(A)), torch.zeros_like(b), ctx.policy_fixed((2, 4, 4, 4))
        took.append(_median(lambda: ctx.solve(mat, b, x, 0.0, 30, pol)))
    assert took[0] < 1.35 * took[1]
