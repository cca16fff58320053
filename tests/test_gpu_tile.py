"""The fp64 product from warp tiles where it can go wrong: fewer rows than a warp or a CTA holds, a
last part of a tile, several tiles per warp, rows that start at odd places, tiles that are just full
(28 nonzeros a row) and matrices just beyond (29, which take the direct loads)."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ALL64 = (4, 4, 4, 4)


@pytest.fixture(scope="module")
def M():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2504_14268_gb300 import mpcg

    return mpcg


def _band(n, half, extra, rng):
    """Symmetric band of half-width `half` (`extra`: every fourth row also holds the entry half + 1
    places on, so that row starts fall on all alignments), strictly dominant diagonal."""
    i = np.arange(n)
    rows, cols, vals = [], [], []
    for k in range(1, half + 1):
        v = rng.uniform(-1, 1, n)
        rows += [i[k:], i[:-k]] if k < n else []
        cols += [i[:-k], i[k:]] if k < n else []
        vals += [v[k:], v[k:]] if k < n else []
    if extra and n > half + 8:
        j = i[(i % 4 == 0) & (i + half + 1 < n)]
        v = rng.uniform(-1, 1, len(j))
        rows += [j, j + half + 1]
        cols += [j + half + 1, j]
        vals += [v, v]
    r = np.concatenate(rows + [i])
    c = np.concatenate(cols + [i])
    v = np.concatenate(vals + [np.full(n, 2.0 * (half + 2))])
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    return n, rp.astype(np.int32), c[o].astype(np.int32), v[o]


@pytest.mark.parametrize("n", [33, 257, 5001, 100003])
@pytest.mark.parametrize("half,extra", [(7, 0), (12, 1), (13, 0), (13, 1), (14, 0)])
def test_product_and_solve(M, n, half, extra):
    rng = np.random.default_rng([n, half, extra])
    A = _band(n, half, extra, rng)
    _, rp, ci, val = A
    x = rng.standard_normal(n)
    ctx = M.Context(0, M.Options(stepped=2, min_k=0))
    mat = ctx.matrix((n, torch.as_tensor(rp).cuda(), torch.as_tensor(ci).cuda(), torch.as_tensor(val).cuda()))
    y = torch.zeros(n, dtype=torch.float64, device="cuda")
    xd = torch.as_tensor(x).cuda()
    ctx.spmv(mat, 4, xd, y)
    ref = np.add.reduceat(val * x[ci], rp[:-1])
    # two summations of at most 31 terms in different orders
    assert np.all(np.abs(y.cpu().numpy() - ref) <= 2 * 31 * 2.0**-53 * np.add.reduceat(np.abs(val * x[ci]), rp[:-1]))
    # eight iterations on a matrix with condition number below (4 half + 6) / 2 <= 31: the rounding
    # errors of each (31 terms a product, log2(n) + 1 levels a dot product) amplified at most so
    sol = torch.zeros_like(y)
    res, _ = ctx.solve(mat, xd, sol, 0.0, 8, ctx.policy_fixed(ALL64))
    want = O.solve(O.Options(min_k=0), A, x, 0.0, 8, fixed=ALL64)
    tol = 8 * 31 * (31 + np.log2(n) + 1) * 2.0**-53 * 8
    assert res["iters"] == want.iters
    assert np.linalg.norm(sol.cpu().numpy() - want.x) <= tol * np.linalg.norm(want.x)
