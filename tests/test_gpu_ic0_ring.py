"""IC(0) solves around the ring of level blocks of the team solver: vectors that stay in global memory
beside a full ring, and grids whose levels do not fit it (other kernels take those). Compared with the
lockstep kernel, which has no ring."""
import numpy as np
import pytest

from paper_2504_14268_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ALL64 = (4, 4, 4, 4)


@pytest.fixture(scope="module")
def M():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2504_14268_gb300 import mpcg

    return mpcg


def _dev(A):
    n, rp, ci, val = A
    return (n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda())


# 2D grid with the vectors in global memory beside a full ring; grids whose levels no longer fit the ring
@pytest.mark.parametrize("A", [I.poisson2d(148), I.fem27_aniso(30, 1e-2), I.fem27_aniso(32, 1e-2),
                               I.diffusion_varcoef((32, 32, 32), 0.5, np.random.default_rng(1))],
                         ids=["2d148", "27pt30", "27pt32", "7pt32"])
def test_ic0_systems_around_the_ring(M, A):
    _, b = I.rhs_from_xstar(A, np.random.default_rng(8))
    out = []
    for mode in (0, 2):
        ctx = M.Context(0, M.Options(min_k=0, precond=2, batch_mode=mode))
        mat = ctx.matrix(_dev(A))
        bd = torch.as_tensor(b).cuda()
        x = torch.zeros_like(bd)
        res = ctx.solve_batched([mat], [bd], [x], [1e-10], [8], ctx.policy_fixed(ALL64))[0]
        out.append((res["outcome"], res["iters"], x.cpu().numpy()))
    assert out[0][:2] == out[1][:2]
    # the substitutions agree bit for bit; fl32(r) may round the other way once sums differ (2^-24)
    assert np.linalg.norm(out[0][2] - out[1][2]) <= 1e-7 * np.linalg.norm(out[1][2])
