"""A graph of team launches may be launched on any stream as soon as it has been created: its tables are
on the device by then, whatever work the creation stream still had."""
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


def test_launch_on_another_stream(M):
    ctx = M.Context(0, M.Options(min_k=0))
    mats, bs = [], []
    for i, m in enumerate((9, 20, 33)):
        A = I.poisson2d(m)
        n, rp, ci, val = A
        mats.append(ctx.matrix((n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda())))
        bs.append(torch.as_tensor(I.rhs_from_xstar(A, np.random.default_rng(i))[1]).cuda())
    pol = ctx.policy_fixed((4, 4, 4, 4))
    xs, ys = [[torch.zeros_like(b) for b in bs] for _ in range(2)]
    want = ctx.solve_batched(mats, bs, ys, [1e-9] * 3, [200] * 3, pol)
    busy, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(100_000_000)  # some 50 ms
    g = ctx.graph(mats, bs, xs, [1e-9] * 3, [200] * 3, pol, stream=busy)
    g.launch(stream=other)
    res = g.results(stream=other)
    for r, w, x, y in zip(res, want, xs, ys):
        assert (r["outcome"], r["iters"]) == (w["outcome"], w["iters"])
        assert torch.equal(x, y)
