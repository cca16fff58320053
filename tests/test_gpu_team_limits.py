"""The team solver at the limits of its forms: rows around a CTA's 512 threads, vectors that stay in
global memory on the whole grid, product tiles of which some exceed their place."""
import numpy as np
import pytest

import oracle as O
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


def _csr(n, r, c, v):
    o = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    return n, rp.astype(np.int32), c[o].astype(np.int32), v[o]


@pytest.mark.parametrize("fmt", [4, 3, 0])
@pytest.mark.parametrize("n", [511, 512, 513])  # one CTA: 7 n - 2 units of work, below 8192
def test_rows_around_one_ctas_threads(M, n, fmt):
    i = np.arange(n)
    r = np.concatenate([i, i[1:], i[:-1]])
    c = np.concatenate([i, i[:-1], i[1:]])
    A = _csr(n, r, c, np.concatenate([np.full(n, 4.0), np.full(2 * n - 2, -1.0)]))
    _, b = I.rhs_from_xstar(A, np.random.default_rng(n))
    f = (fmt, 4, 4, 4)
    ctx = M.Context(0, M.Options(min_k=0))
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    res, hist = ctx.solve(ctx.matrix(_dev(A)), torch.as_tensor(b).cuda(), x, 0.0, 6, ctx.policy_fixed(f), history_cap=6)
    ref = O.solve(O.Options(min_k=0), A, b, 0.0, 6, fixed=f)
    assert res["iters"] == ref.iters == 6
    # six iterations on a matrix of condition 3: sums of 513 terms in another order; fp32 rows of three
    # terms rounded after each (6 * 3 * 3 * 2^-24); an fp16 rounding of p that falls the other way moves
    # one of 513 terms by 2^-11
    tol = {4: 1e-12, 3: 4e-6, 0: 1e-4}[fmt]
    assert np.abs(hist["nu"] / ref.hist["nu"] - 1).max() <= tol
    assert np.linalg.norm(x.cpu().numpy() - ref.x) <= tol * np.linalg.norm(ref.x)


@pytest.mark.parametrize("true_every", [0, 3])
@pytest.mark.parametrize("pol", [ALL64, (3, 4, 4, 4)])
def test_whole_grid_with_vectors_in_global_memory(M, pol, true_every):
    """1090^2 rows: some 7,800 a CTA, 250 KB of vectors. Against the stepped kernels; nine iterations
    from sums of 1.2e6 terms in other orders."""
    A = I.poisson2d(1090)
    b = np.random.default_rng(2).uniform(-1, 1, A[0])
    out = []
    for stepped in (1, 2):
        ctx = M.Context(0, M.Options(min_k=0, stepped=stepped, true_res_every=true_every))
        x = torch.zeros(A[0], dtype=torch.float64, device="cuda")
        res, _ = ctx.solve(ctx.matrix(_dev(A)), torch.as_tensor(b).cuda(), x, 0.0, 9, ctx.policy_fixed(pol))
        out.append((res, x.cpu().numpy()))
    (r0, x0), (r1, x1) = out
    assert r0["kernel_launches"] == 1 and r1["kernel_launches"] > 1
    for key in ("outcome", "iters", "n_true_checks"):
        assert r0[key] == r1[key]
    tol = 1e-11 if pol == ALL64 else 1e-5  # (fp32: roundings of p that fall the other way)
    assert np.linalg.norm(x0 - x1) <= tol * np.linalg.norm(x1)
    assert abs(r0["rel_res_true"] / r1["rel_res_true"] - 1) <= tol


def _uneven(n):
    """Every 32 consecutive rows hold 880 entries (a matrix for tiles of 896), 768 of them in 16 rows
    (above the 592 of an fp64 tile of 16 rows)."""
    i = np.arange(n)
    heavy = i % 32 < 16
    rows, cols = [], []
    for d in range(-44, 45):
        j = i + d
        ok = (j >= 0) & (j < n)
        ok[ok] &= (abs(d) <= 3) | (heavy[i[ok]] & heavy[j[ok]])
        rows.append(i[ok])
        cols.append(j[ok])
    r, c = np.concatenate(rows), np.concatenate(cols)
    rng = np.random.default_rng(7)
    w = rng.uniform(-1, 1, n)
    return _csr(n, r, c, np.where(r == c, 60.0, w[r] * w[c]))


@pytest.mark.parametrize("fmt", [4, 3, 2, 1])
def test_tiles_that_exceed_their_place(M, fmt):
    """One iteration on the whole grid: nu against the oracle's (a product differs by at most one unit
    of its format, fp32 by its accumulation bound of 48 terms)."""
    A = _uneven(150_000)
    lens = np.diff(A[1])
    win = np.convolve(lens, np.ones(32, int), "valid")
    assert win.max() == 880 and np.add.reduceat(lens, np.arange(64, 1000, 32)).min() > 592
    b = np.random.default_rng(3).uniform(-1, 1, A[0])
    f = (fmt, 4, 4, 4)
    ctx = M.Context(0, M.Options(min_k=0))
    x = torch.zeros(A[0], dtype=torch.float64, device="cuda")
    _, hist = ctx.solve(ctx.matrix(_dev(A)), torch.as_tensor(b).cuda(), x, 0.0, 1, ctx.policy_fixed(f), history_cap=1)
    ref = O.solve(O.Options(min_k=0), A, b, 0.0, 1, fixed=f)
    assert abs(hist["nu"][0] / ref.hist["nu"][0] - 1) <= {3: 2 * 48 * 2.0**-24, 4: 1e-13}.get(fmt, 1e-12)
