"""The team solver (one system per cluster of CTAs, or on the whole grid) where its splits can go
wrong: sizes around warps, CTAs and the switch from a cluster to the grid; rows around the lengths
at which a warp or the CTA sums them; systems that share a cluster; the short scalar step against
the full one (a history forces the latter); IC(0) substitutions around the 32-row groups of a
level. Compared with the oracle's fp64 solve, or with the lockstep kernel's solve of the same
systems (batch_mode 2), whose sums run in another order."""
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


def _solve(M, ctx, A, b, pol, tol, cap, **kw):
    bd = torch.as_tensor(b).cuda()
    x = torch.zeros_like(bd)
    res, hist = ctx.solve(ctx.matrix(_dev(A)), bd, x, tol, cap, pol, **kw)
    return res, hist, x.cpu().numpy()


# 1 row; warp edges (31-33 rows: 5.6^2); one CTA's 1024 threads (32^2, 33^2); a cluster's several
# rows per thread; nnz + 4 n on both sides of the 160,000 from which the grid solves it (133^2, 134^2)
@pytest.mark.parametrize("m", [1, 2, 5, 6, 31, 32, 33, 57, 90, 133, 134, 181])
def test_sizes_against_the_oracle(M, m):
    A = I.poisson2d(m) if m > 1 else (1, np.array([0, 1], np.int32), np.array([0], np.int32), np.array([4.0]))
    xs, b = I.rhs_from_xstar(A, np.random.default_rng(m))
    ctx = M.Context(0, M.Options(min_k=0))
    res, _, x = _solve(M, ctx, A, b, ctx.policy_fixed(ALL64), 1e-10, 2000)
    ref = O.solve(O.Options(min_k=0), A, b, 1e-10, 2000, fixed=ALL64)
    assert res["outcome"] == ref.outcome == O.CONVERGED
    assert abs(res["iters"] - ref.iters) <= 1  # (a count moves by one when rho lands beside tol)
    # both stop below 1e-10 of the residual: errors of the same size
    assert np.linalg.norm(x - xs) <= 10 * np.linalg.norm(ref.x - xs) + 1e-14 * np.linalg.norm(xs)


@pytest.mark.parametrize("n", [6000, 40000])  # a cluster, the grid
@pytest.mark.parametrize("fmt", range(8))
def test_row_lengths_around_the_splits(M, fmt, n):
    """One iteration on a ring with hub rows of 32..34, 511..514 and 1023..1026 nonzeros:
    nu = p^T fl(A fl(p)) against the oracle's. Each q_i differs by at most one unit of its format
    (fp32: its accumulation bound of 1026 terms), and nu's relative error is that of q's largest."""
    rng = np.random.default_rng(5)
    lens = [32, 33, 34, 511, 512, 513, 514, 1023, 1024, 1025, 1026]
    rows = [dict() for _ in range(n)]
    for i in range(n):
        rows[i][i] = 3.0
        for j in ((i + 1) % n, (i - 1) % n):
            rows[i][j] = -1.0
    hubs = list(range(100, 100 + n // 12 * len(lens), n // 12))
    for h, ln in zip(hubs, lens):
        for j in rng.choice(np.arange(n), size=ln + 40, replace=False):
            j = int(j)
            if len(rows[h]) >= ln:
                break
            if j in rows[h] or j in hubs:
                continue
            rows[h][j] = rows[j][h] = -0.5
        rows[h][h] = 0.5 * ln + 3.0
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    ci = np.concatenate([sorted(r) for r in rows]).astype(np.int32)
    val = np.concatenate([[r[c] for c in sorted(r)] for r in rows])
    A = (n, rp, ci, val)
    assert sorted(np.diff(rp)[hubs]) == lens
    b = rng.uniform(-1, 1, n)
    f = (fmt, 4, 4, 4)
    ctx = M.Context(0, M.Options(min_k=0))
    _, hist, _ = _solve(M, ctx, A, b, ctx.policy_fixed(f), 1e-12, 1, history_cap=1)
    ref = O.solve(O.Options(min_k=0), A, b, 1e-12, 1, fixed=f)
    tol = {3: 2 * 1026 * 2.0 ** -24, 4: 1e-13}.get(fmt, 1e-12)  # the other products are correctly rounded
    assert abs(hist["nu"][0] / ref.hist["nu"][0] - 1) <= tol


@pytest.mark.parametrize("fmts", [ALL64, (2, 4, 4, 4), (1, 4, 4, 4)])
def test_systems_sharing_clusters(M, fmts):
    """Eleven systems from 1 to 9000 rows in one launch, against the lockstep kernel."""
    sets = [I.poisson2d(m) for m in (2, 3, 6, 11, 20, 33, 50, 70, 95)]
    sets += [I.fem27_aniso(9, 1e-2), (1, np.array([0, 1], np.int32), np.array([0], np.int32), np.array([2.0]))]
    bs = [I.rhs_from_xstar(A, np.random.default_rng(i))[1] for i, A in enumerate(sets)]
    out = []
    for mode in (0, 2):
        ctx = M.Context(0, M.Options(min_k=0, batch_mode=mode))
        mats = [ctx.matrix(_dev(A)) for A in sets]
        bd = [torch.as_tensor(b).cuda() for b in bs]
        x = [torch.zeros_like(b) for b in bd]
        res = ctx.solve_batched(mats, bd, x, [1e-9] * len(sets), [25] * len(sets), ctx.policy_fixed(fmts))
        out.append((res, [v.cpu().numpy() for v in x]))
    for r0, r1, x0, x1 in zip(out[0][0], out[1][0], out[0][1], out[1][1]):
        assert (r0["outcome"], r0["iters"]) == (r1["outcome"], r1["iters"])
        # 25 iterations from sums that differ in their last bits
        assert np.linalg.norm(x0 - x1) <= 1e-9 * np.linalg.norm(x1) + 1e-300


@pytest.mark.parametrize("kind", ["fixed", "schedule", "table"])
@pytest.mark.parametrize("m", [20, 140])
def test_short_step_equals_full_step(M, kind, m):
    """Without a history the short scalar step runs, with one the full step: the same bits in x, the
    same counts and decisions (the table changes formats at bin edges, tol stops the solve)."""
    A = I.poisson2d(m)
    _, b = I.rhs_from_xstar(A, np.random.default_rng(3))
    ctx = M.Context(0, M.Options())
    if kind == "fixed":
        pol = ctx.policy_fixed((2, 4, 4, 4))
    elif kind == "schedule":
        pol = ctx.policy_schedule([(2, 4, 3, 3)] * 7 + [(1, 2, 4, 4)] * 5 + [ALL64])
    else:
        Q = np.zeros((4, 100, 5))
        for s in range(100):
            for op in range(4):
                Q[op, s, (1, 2, 3, 4, 4, 4, 4, 4, 4, 4)[s % 10]] = 1.0
        pol = ctx.policy_qtable(Q)
    r0, _, x0 = _solve(M, ctx, A, b, pol, 1e-6, 400)
    r1, hist, x1 = _solve(M, ctx, A, b, pol, 1e-6, 400, history_cap=400)
    assert np.array_equal(x0, x1)
    for key in ("outcome", "iters", "near_edge_count", "rel_res_rec", "rel_res_true"):
        assert r0[key] == r1[key], key
    assert np.array_equal(r0["action_hist"], r1["action_hist"])
    assert np.array_equal(hist["k"][: r1["iters"]], np.arange(r1["iters"]))


# levels of one row, of 31..33 and 64..66 rows (2D grids: the widest level has m rows), 27-point rows
@pytest.mark.parametrize("A", [I.poisson2d(2), I.poisson2d(31), I.poisson2d(33), I.poisson2d(65), I.fem27_aniso(9, 1e-2),
                               I.banded_spd(900, 11, 1.0, np.random.default_rng(2))], ids=lambda A: f"n{A[0]}")
def test_ic0_levels(M, A):
    _, b = I.rhs_from_xstar(A, np.random.default_rng(8))
    out = []
    for mode in (0, 2):
        ctx = M.Context(0, M.Options(min_k=0, precond=2, batch_mode=mode))
        mat = ctx.matrix(_dev(A))
        bd = torch.as_tensor(b).cuda()
        x = torch.zeros_like(bd)
        res = ctx.solve_batched([mat], [bd], [x], [1e-10], [12], ctx.policy_fixed(ALL64))[0]
        out.append((res["outcome"], res["iters"], x.cpu().numpy()))
    assert out[0][:2] == out[1][:2]
    # the substitutions agree bit for bit; fl32(r) may round the other way once sums differ (2^-24)
    assert np.linalg.norm(out[0][2] - out[1][2]) <= 1e-7 * np.linalg.norm(out[1][2]) + 1e-300
