"""Table-driven IC(0) solves of the sizes at which the ring of level blocks, the vector and the table
together nearly fill a CTA's shared memory, against the lockstep kernel."""
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


@pytest.mark.parametrize("bins", [(10, 10), (24, 10), (64, 16)])  # tables of 16 and 38 KB, and one that is not held
@pytest.mark.parametrize("m", [22, 27])
def test_table_beside_the_ring(M, m, bins):
    A = I.fem27_aniso(m, 1e-2)
    n, rp, ci, val = A
    _, b = I.rhs_from_xstar(A, np.random.default_rng(m))
    S = bins[0] * bins[1]
    Q = np.zeros((4, S, 5))
    Q[1:, :, 4] = 1.0
    Q[0, :, 3], Q[0, np.arange(S) % bins[1] > 1, 4] = 0.5, 1.0  # fp32 products while the residual is large
    out = []
    for mode in (0, 2):
        ctx = M.Context(0, M.Options(min_k=0, precond=2, batch_mode=mode, b_bins=bins[0], r_bins=bins[1]))
        mat = ctx.matrix((n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda()))
        bd = torch.as_tensor(b).cuda()
        x = torch.zeros_like(bd)
        res = ctx.solve_batched([mat], [bd], [x], [1e-10], [10], ctx.policy_qtable(Q, np.ones((4, S), np.int32)))[0]
        out.append((res, x.cpu().numpy()))
    (r0, x0), (r1, x1) = out
    assert (r0["outcome"], r0["iters"]) == (r1["outcome"], r1["iters"])
    assert np.array_equal(r0["action_hist"], r1["action_hist"])
    # fl32(r) and fp32 roundings of p may fall the other way once sums differ (2^-24), ten iterations
    assert np.linalg.norm(x0 - x1) <= 1e-6 * np.linalg.norm(x1)
