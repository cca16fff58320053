"""Performance cases of the mixed-precision CG library, through its Python binding.

A case is what a program that uses the library asks of it: one solve of one system (small
ones, where launches and the scalar steps between phases count, up to grids that stream HBM), a
batch of uneven systems replayed as a graph, batches and single systems with the IC(0)
preconditioner, rounds of Q-learning, the fitting of the network, and the product alone.
The families are those of `paper_2504_14268_gb300/inputs.py`, built here on the GPU where the
host would take long.

Solves run to a relative residual of 1e-8 or to the iteration budget of the case; the budgets
mostly lie below the count that 1e-8 takes. Families on which plain CG multiplies rounding
errors from one iteration to the next (high-contrast diffusion, power-law graphs) are solved with
the Jacobi preconditioner, as one would; large systems with a low-precision product get short
budgets, since one rounding that falls the other way is multiplied in the same way.
"""
import math

import numpy as np
import torch

from paper_2504_14268_gb300 import inputs as I
from paper_2504_14268_gb300 import mpcg as M

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F = {"fp16": 0, "bf16": 1, "tf32": 2, "fp32": 3, "fp64": 4, "bf16r": 5, "fp16r": 6, "q52": 7}
SIZE = {"fp16": 2, "bf16": 2, "tf32": 4, "fp32": 4, "fp64": 8, "bf16r": 2, "fp16r": 2, "q52": 1}
PARAM = {0: (11, -14, 15), 1: (8, -126, 127), 2: (11, -126, 127), 3: (24, -126, 127), 7: (3, -14, 15)}
TOL = 1e-8


# ---------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------

def listed():
    return [
        # the paper's smallest system: everything between two phases is latency
        dict(name="poisson32_fp64", kind="solve", family="poisson2d", m=32, precond=0, policy="fp64,fp64,fp64,fp64",
             iters=80, host=False),
        # one system of Section 5.2 from host buffers, a table that starts cheap and ends in fp64
        dict(name="subdomain80_table", kind="solve", family="subdomain", m=80, precond=0, policy="table:tf32",
             iters=150, host=True),
        # a system of the training family (7-point, odd edge), Jacobi, tf32 product
        dict(name="diffusion37_tf32", kind="solve", family="diffusion3", m=37, precond=1,
             policy="tf32,fp64,fp64,fp64", iters=60, host=False),
        # a power-law graph Laplacian: rows from 6 to thousands of nonzeros, fp64
        dict(name="graph160k_fp64", kind="solve", family="graph", m=160000, precond=1, policy="fp64,fp64,fp64,fp64",
             iters=16, host=False),
        # the middle of the FEM family: the matrix still fits the L2
        dict(name="fem64_table", kind="solve", family="fem27", m=64, precond=0, policy="table:tf32", iters=24,
             host=False),
        # the large single solve, HBM streams the matrix every iteration: the table of the {fp32, fp64} set
        dict(name="fem160_table", kind="solve", family="fem27", m=160, precond=0, policy="table:fp32", iters=16,
             host=False),
        # ... and all of it in fp64, an edge that is no multiple of anything
        dict(name="fem143_fp64", kind="solve", family="fem27", m=143, precond=0, policy="fp64,fp64,fp64,fp64", iters=60,
             host=False),
        # uneven systems (2D and 3D diffusion, banded) in one batch, replayed as a graph
        dict(name="batch48_fp64", kind="batch", count=48, n_lo=1000, n_hi=60000, policy="fp64,fp64,fp64,fp64", iters=60),
        # the paper's protocol: its Poisson systems with the fp32 IC(0) preconditioner in a batch
        dict(name="ic_batch24", kind="ic_batch", m=80, count=24, iters=40),
        # one larger system with IC(0): the substitutions' dependency chains
        dict(name="ic_fem28", kind="solve", family="fem27", m=28, precond=2, policy="fp64,fp64,fp64,fp64", iters=20,
             host=False),
        # rounds of Algorithm 1 on small FEM systems, every format explored
        dict(name="train8", kind="train", count=8, m_lo=16, m_hi=30, episodes=2, iters=24),
        # the network's fitted-Q steps at the batch that the graph evaluation uses
        dict(name="mlp1024", kind="mlp", count=20000, steps=40, batch=1024, hidden=64),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges (sizes log-uniform; each no larger than the largest listed)."""
    kind = rng.choice(["poisson2d", "subdomain", "diffusion3", "graph", "fem27", "fem27", "fem27", "spmv", "batch",
                       "ic_batch", "ic", "train", "mlp"])
    stable = ["fp64,fp64,fp64,fp64", "tf32,fp64,fp64,fp64", "bf16,fp64,fp64,fp64", "fp16r,fp64,fp64,fp64"]
    if kind == "poisson2d":
        return dict(kind="solve", family=kind, m=int(_log(rng, 16, 300)), precond=rng.choice([0, 1]),
                    policy=rng.choice(stable), iters=rng.randint(30, 60), host=rng.random() < 0.5)
    if kind == "subdomain":
        return dict(kind="solve", family=kind, m=int(_log(rng, 40, 200)), precond=0, policy="table:tf32",
                    iters=rng.randint(50, 110), host=True)
    if kind == "diffusion3":
        return dict(kind="solve", family=kind, m=int(_log(rng, 12, 90)), precond=1,
                    policy=rng.choice(["fp64,fp64,fp64,fp64", "tf32,fp64,fp64,fp64"]), iters=rng.randint(20, 40),
                    host=False)
    if kind == "graph":
        return dict(kind="solve", family=kind, m=int(_log(rng, 8000, 400000)), precond=1,
                    policy="fp64,fp64,fp64,fp64", iters=rng.randint(12, 16), host=False)
    if kind == "fem27":
        m = int(_log(rng, 20, 140))
        pol = rng.choice(list(stable) + ["fp32,fp64,fp32,fp64", "table:fp32"])
        return dict(kind="solve", family=kind, m=m, precond=0, policy=pol,
                    iters=rng.randint(10, 14) if "fp32" in pol else rng.randint(20, 24 if m > 50 else 58),
                    host=False)
    if kind == "spmv":
        return dict(kind="spmv", family=rng.choice(["fem27", "diffusion3", "graph"]), m=int(_log(rng, 20, 140)),
                    formats=",".join(rng.sample(["fp64", "fp32", "tf32", "bf16", "fp16", "fp16r", "bf16r", "q52"], 3)))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(5, 48), n_lo=1000, n_hi=int(_log(rng, 4000, 60000)),
                    policy=rng.choice(["fp64,fp64,fp64,fp64", "tf32,fp64,fp64,fp64"]), iters=rng.randint(20, 60))
    if kind == "ic_batch":
        return dict(kind="ic_batch", m=rng.randint(30, 90), count=rng.randint(4, 24), iters=rng.randint(15, 30))
    if kind == "ic":
        return dict(kind="solve", family=rng.choice(["fem27", "poisson2d"]), m=rng.randint(16, 28), precond=2,
                    policy="fp64,fp64,fp64,fp64", iters=rng.randint(10, 18), host=False)
    if kind == "train":
        return dict(kind="train", count=rng.randint(2, 8), m_lo=12, m_hi=rng.randint(16, 28), episodes=2,
                    iters=rng.randint(12, 24))
    return dict(kind="mlp", count=rng.randint(3000, 20000), steps=rng.randint(10, 40),
                batch=int(_log(rng, 64, 1024)), hidden=rng.choice([32, 48, 64, 96]))


# ---------------------------------------------------------------------------------------
# Matrices (CSR on the GPU: (n, row_ptr int32, col int32, val float64))
# ---------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _csr_from_slots(col, val, ok):
    """CSR of per-row slots in increasing column order ([n][slots], ok marks the stored ones)."""
    n = col.shape[0]
    rp = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rp[1:] = ok.sum(1).cumsum(0).to(torch.int32)
    return n, rp, col[ok].to(torch.int32).contiguous(), val[ok].contiguous()


def _fem27(N, eps):
    kc, mc = (-1.0, 2.0, -1.0), (1 / 6, 4 / 6, 1 / 6)
    n = N ** 3
    row = torch.arange(n, device=DEV, dtype=torch.int32)
    ijk = (row // (N * N), row // N % N, row % N)
    col = torch.empty(n, 27, dtype=torch.int32, device=DEV)
    ok = torch.empty(n, 27, dtype=torch.bool, device=DEV)
    coef = []
    for t in range(27):
        d = (t // 9 - 1, t // 3 % 3 - 1, t % 3 - 1)
        a = [c + s for c, s in zip(ijk, d)]
        ok[:, t] = (a[0] >= 0) & (a[0] < N) & (a[1] >= 0) & (a[1] < N) & (a[2] >= 0) & (a[2] < N)
        col[:, t] = row + (d[0] * N + d[1]) * N + d[2]
        x, y, z = (s + 1 for s in d)
        coef.append(kc[x] * mc[y] * mc[z] + mc[x] * kc[y] * mc[z] + eps * mc[x] * mc[y] * kc[z])
    val = torch.tensor(coef, dtype=torch.float64, device=DEV).expand(n, 27)
    return _csr_from_slots(col, val, ok)


def _diffusion(shape, sigma, g):
    """Cell-centred 5- or 7-point diffusion, log-normal cells, harmonic-mean faces, Dirichlet."""
    d, n = len(shape), int(np.prod(shape))
    kap = torch.exp(sigma * _randn(g, *shape))
    row = torch.arange(n, device=DEV, dtype=torch.int64).reshape(shape)
    diag = torch.zeros_like(kap)
    lower, upper = [], []
    for ax in range(d):
        step = int(np.prod(shape[ax + 1:]))
        face = torch.zeros_like(kap)  # face above each cell along ax
        k = shape[ax]
        if k > 1:
            a, b = kap.narrow(ax, 0, k - 1), kap.narrow(ax, 1, k - 1)
            f = 2.0 * a * b / (a + b)
            face.narrow(ax, 0, k - 1).copy_(f)
            diag.narrow(ax, 0, k - 1).add_(f)
            diag.narrow(ax, 1, k - 1).add_(f)
        diag.narrow(ax, 0, 1).add_(2.0 * kap.narrow(ax, 0, 1))
        diag.narrow(ax, k - 1, 1).add_(2.0 * kap.narrow(ax, k - 1, 1))
        below = torch.zeros_like(face)
        if k > 1:
            below.narrow(ax, 1, k - 1).copy_(face.narrow(ax, 0, k - 1))
        lower.append((row - step, -below))
        upper.append((row + step, -face))
    slots = lower + [(row, diag)] + upper[::-1]
    col = torch.stack([c.reshape(-1) for c, _ in slots], 1)
    val = torch.stack([v.reshape(-1) for _, v in slots], 1)
    return _csr_from_slots(col, val, val != 0)


def _banded(n, kd, lam, g):
    """L L^T + lam I, L lower triangular with half-bandwidth kd and N(0, 1) entries."""
    ab = _randn(g, kd + 1, n)
    i = torch.arange(n, device=DEV)
    for m in range(1, kd + 1):
        ab[m, :m] = 0.0
    diags = torch.zeros(kd + 1, n, dtype=torch.float64, device=DEV)  # entry (i, i - d)
    for d in range(kd + 1):
        diags[d, d:] = (ab[d:, d:] * ab[: kd + 1 - d, : n - d]).sum(0)
    diags[0] += lam
    offs = torch.arange(-kd, kd + 1, device=DEV)
    col = i[:, None] + offs[None, :]
    ok = (col >= 0) & (col < n)
    hi = torch.maximum(i[:, None].expand_as(col), col).clamp(0, n - 1)
    val = diags[offs.abs()[None, :].expand_as(col), hi]
    return _csr_from_slots(col, val, ok)


def _graph(n, g, m=6, shift=1e-4):
    """Shifted Laplacian of a power-law graph: node v joins m earlier nodes floor(v u^2), the
    degree profile of preferential attachment (degree of node i ~ i^-1/2)."""
    v = torch.arange(1, n, device=DEV).repeat_interleave(m)
    w = (v * _rand(g, v.numel()) ** 2).to(torch.int64)
    key = torch.unique(torch.cat([v * n + w, w * n + v]))
    r, c = key // n, key % n
    deg = torch.bincount(r, minlength=n)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = (deg + 1).cumsum(0)
    # each row: columns below the diagonal, the diagonal, columns above
    below = torch.bincount(r[c < r], minlength=n)
    pos = torch.arange(key.numel(), device=DEV) + r + (c > r)
    col = torch.empty(key.numel() + n, dtype=torch.int32, device=DEV)
    val = torch.full((key.numel() + n,), -1.0, dtype=torch.float64, device=DEV)
    col[pos] = c.to(torch.int32)
    dp = rp[:-1] + below
    col[dp] = torch.arange(n, device=DEV, dtype=torch.int32)
    val[dp] = deg.to(torch.float64) + shift
    return n, rp.to(torch.int32), col, val


def _matvec(A, val, x):
    n, rp, ci, _ = A
    return torch.sparse_csr_tensor(rp, ci, val, (n, n), dtype=torch.float64) @ x


def _rhs(A, g):
    xs = 2.0 * _rand(g, A[0]) - 1.0
    return _matvec(A, A[3], xs), xs


def _system(family, m, seed):
    """(matrix, right-hand side) of a family; m: grid edge (graph: number of nodes)."""
    g = _gen(seed)
    if family == "subdomain":
        (n, rp, ci, val), b = I.poisson_subdomain(int(seed) % (1 << 31), m)
        dev = [torch.as_tensor(v).to(DEV) for v in (rp, ci, val)]
        return (n, *dev), torch.as_tensor(b).to(DEV)
    if family == "poisson2d":
        A = _diffusion((m, m), 0.0, g)
        A[3][A[3] > 0] = 4.0
    elif family == "diffusion3":
        A = _diffusion((m, m, m), 1.0, g)
    elif family == "fem27":
        A = _fem27(m, 1e-3)
    else:
        A = _graph(m, g)
    return A, _rhs(A, g)[0]


def _nnz(family, m):
    """(rows, nonzeros) of a family, for the work of a case."""
    if family in ("poisson2d", "subdomain"):
        return m * m, 5 * m * m - 4 * m
    if family == "diffusion3":
        return m ** 3, 7 * m ** 3 - 6 * m * m
    if family == "fem27":
        return m ** 3, (3 * m - 2) ** 3
    return m, 13 * m


def _graph_nodes(case):
    return case["m"] if case.get("kind") != "spmv" else case["m"] ** 2 * 10  # a graph of the grids' size


# ---------------------------------------------------------------------------------------
# Policies
# ---------------------------------------------------------------------------------------

def _table(kind):
    """A Q-table as training leaves it: one format per operation and residual bin (delta = 1.6
    decades), cheap while the residual is large."""
    low, top = F[kind], F["fp64"]
    Q = np.zeros((4, 100, 5))
    for s in range(100):
        j = s % 10
        pick = (low if j <= 2 else top, low if j == 0 and kind == "tf32" else top, top, top)
        for op in range(4):
            Q[op, s, pick[op]] = 1.0
    return Q


def _policy(ctx, text):
    if text.startswith("table:"):
        return ctx.policy_qtable(_table(text[6:]))
    return ctx.policy_fixed([F[t] for t in text.split(",")])


def _formats(text):
    """k, rho -> the four formats (the state of Section 4.1 for a table)."""
    if not text.startswith("table:"):
        fixed = [F[t] for t in text.split(",")]
        return lambda k, rho: fixed
    best = _table(text[6:]).argmax(2)
    return lambda k, rho: [int(a) for a in best[:, _state(k, rho)]]


def _state(k, rho):
    return min(k // 100, 9) * 10 + sum(rho <= 10.0 ** (-1.6 * m) for m in range(1, 10))


# ---------------------------------------------------------------------------------------
# prepare, run
# ---------------------------------------------------------------------------------------

def _batch_systems(case, seed):
    """Thirds of 2D diffusion, 3D diffusion and banded systems, n log-uniform."""
    r = np.random.default_rng([int(seed), 4])
    out = []
    for i in range(case["count"]):
        sizes = np.random.default_rng([i, 4])  # the sizes of a batch are the case's own
        n = int(round(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        kd = int(sizes.integers(5, 65))
        g = _gen(int(r.integers(1 << 62)))
        if i % 3 == 0:
            e = int(round(math.sqrt(n)))
            A, cap = _diffusion((e, e), 1.0, g), case["iters"]
        elif i % 3 == 1:
            e = int(round(n ** (1 / 3)))
            A, cap = _diffusion((e, e, e), 1.0, g), case["iters"]
        else:  # plain CG loses its digits on these within some 25 iterations: a short budget
            A, cap = _banded(n, min(kd, n - 1), 1e-2, g), 12
        out.append((A, _rhs(A, g)[0], cap))
    return out


def _ic_systems(case, seed):
    return [(*_system("subdomain", case["m"], int(seed) * 101 + i), case["iters"]) for i in range(case["count"])]


def _train_systems(case, seed):
    edges = np.linspace(case["m_lo"], case["m_hi"], case["count"]).astype(int)
    out = []
    for i, m in enumerate(edges):
        A = _fem27(int(m), (1e-3, 3e-3, 1e-2)[i % 3])
        out.append((A, _rhs(A, _gen(int(seed) * 37 + i))[0]))
    return out


def _transitions(case, seed):
    """Transitions of the kind an episode leaves: features of order one, log-residual rewards."""
    r = np.random.default_rng([int(seed), 7])
    d = np.zeros(case["count"], dtype=M.TRANS_DTYPE)
    d["f"] = (0.5 * r.standard_normal((case["count"], 16))).astype(np.float32)
    d["f_next"] = (d["f"] + 0.1 * r.standard_normal((case["count"], 16))).astype(np.float32)
    d["act"] = r.integers(0, 5, (case["count"], 4))
    d["reward"] = r.uniform(0.0, 8.0, case["count"])
    d["done"] = r.random(case["count"]) < 0.01
    w = (0.1 * r.standard_normal(M.mlp_nparams(case["hidden"], 5))).astype(np.float32)
    return d, w


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "solve":
        ctx = M.Context(0, M.Options(precond=case["precond"]))
        A, b = _system(case["family"], case["m"], seed)
        st.update(ctx=ctx, mat=ctx.matrix(A), pol=_policy(ctx, case["policy"]))
        if case["precond"] == 2:
            st["mat"].ic0()
        if case["host"]:
            st.update(b=b.cpu().numpy(), x=np.zeros(A[0]))
        else:
            st.update(b=b, x=torch.zeros_like(b))
    elif kind == "spmv":
        ctx = M.Context(0)
        m = _graph_nodes(case) if case["family"] == "graph" else case["m"]
        A, b = _system(case["family"], m, seed)
        fm = [F[t] for t in case["formats"].split(",")]
        st.update(ctx=ctx, mat=ctx.matrix(A), b=b, formats=fm, ys=[torch.zeros_like(b) for _ in fm])
    elif kind in ("batch", "ic_batch"):
        ctx = M.Context(0, M.Options(precond=2 if kind == "ic_batch" else 1))
        sysm = _ic_systems(case, seed) if kind == "ic_batch" else _batch_systems(case, seed)
        x = torch.zeros(sum(A[0] for A, _, _ in sysm), dtype=torch.float64, device=DEV)
        xs = list(torch.split(x, [A[0] for A, _, _ in sysm]))
        args = ([ctx.matrix(A) for A, _, _ in sysm], [b for _, b, _ in sysm], xs, [TOL] * len(sysm),
                [cap for _, _, cap in sysm], _policy(ctx, case.get("policy", "fp64,fp64,fp64,fp64")))
        if kind == "ic_batch":
            for m in args[0]:
                m.ic0()
        st.update(ctx=ctx, args=args, x=x, graph=ctx.graph(*args) if kind == "batch" else None)
    elif kind == "train":
        ctx = M.Context(0, M.Options(seed=int(seed) % 1000))
        sysm = _train_systems(case, seed)
        st.update(ctx=ctx, mats=[ctx.matrix(A) for A, _ in sysm], bs=[b for _, b in sysm])
    else:
        d, w = _transitions(case, seed)
        st.update(ctx=M.Context(0, M.Options(mlp_hidden=case["hidden"])), data=d, w=w)
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "solve":
        res, _ = ctx.solve(st["mat"], st["b"], st["x"], TOL, case["iters"], st["pol"])
        return {"x": st["x"], "iters": res["iters"], "outcome": res["outcome"], "actions": res["action_hist"]}
    if kind == "spmv":
        for f, y in zip(st["formats"], st["ys"]):
            ctx.spmv(st["mat"], f, st["b"], y)
        return st["ys"]
    if kind == "batch":
        st["graph"].launch()
        res = st["graph"].results()
    elif kind == "ic_batch":
        res = ctx.solve_batched(*st["args"])
    if kind in ("batch", "ic_batch"):
        return {"x": st["x"], "iters": np.array([r["iters"] for r in res])}
    if kind == "train":  # a new table each pass: training updates it in place
        pol = ctx.policy_qtable(np.zeros((4, 100, 5)), np.zeros((4, 100), dtype=np.int32))
        its = ctx.train_qtable(st["mats"], st["bs"], TOL, case["iters"], case["episodes"], pol, want_iters=True)
        Q, visits = pol.qtable()
        return {"Q": Q, "visits": visits, "iters": its}
    pol = ctx.policy_mlp(st["w"])
    loss = ctx.mlp_train(pol, st["data"], case["steps"], case["batch"], target_sync=20, seed=3)
    return {"params": pol.mlp_params(), "loss": loss}


# ---------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------

def _iteration(n, nnz, fmt, precond):
    """Bytes and operations of one iteration with each array touched once: the product (values,
    columns, row pointers, p in its format, q), r (read, written), x and p (read, written)."""
    v = SIZE[fmt]
    by = nnz * (v + 4) + 4 * n + 2 * n * v + 16 * n + 32 * n
    fl = 2 * nnz + 10 * n
    if precond == 1:
        by += 8 * n
    if precond == 2:  # both substitutions: the factor (fp32) and its columns
        by += nnz * 8 + 16 * n
        fl += 2 * nnz
    return by, fl


def work(case):
    kind = case["kind"]
    if kind == "solve":
        n, z = _nnz(case["family"], case["m"])
        fmt = case["policy"][6:] if case["policy"].startswith("table:") else case["policy"].split(",")[0]
        by, fl = _iteration(n, z, fmt, case["precond"])
        return {"bytes": case["iters"] * by + 40 * n, "flops": case["iters"] * fl}
    if kind == "spmv":
        n, z = _nnz(case["family"], _graph_nodes(case) if case["family"] == "graph" else case["m"])
        fm = case["formats"].split(",")
        return {"bytes": sum(z * (SIZE[f] + 4) + 4 * n + 16 * n for f in fm), "flops": 2 * z * len(fm)}
    if kind == "batch":
        by = fl = 0
        for i in range(case["count"]):
            sizes = np.random.default_rng([i, 4])
            n = int(round(math.exp(sizes.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
            z, cap = ((5, case["iters"]), (7, case["iters"]), (2 * int(sizes.integers(5, 65)) + 1, 12))[i % 3]
            one = _iteration(n, n * z, case["policy"].split(",")[0], 1)
            by, fl = by + cap * one[0], fl + cap * one[1]
        return {"bytes": by, "flops": fl}
    if kind == "ic_batch":
        by, fl = _iteration(*_nnz("subdomain", case["m"]), "fp64", 2)
        return {"bytes": case["count"] * case["iters"] * by, "flops": case["count"] * case["iters"] * fl}
    if kind == "train":
        by = fl = 0
        for m in np.linspace(case["m_lo"], case["m_hi"], case["count"]).astype(int):
            one = _iteration(*_nnz("fem27", int(m)), "fp32", 0)
            by, fl = by + one[0], fl + one[1]
        k = case["episodes"] * case["iters"]
        return {"bytes": k * by, "flops": k * fl}
    h = case["hidden"]
    npar = 16 * h + h + h * h + h + 20 * h + 20
    by = case["count"] * 152 + case["steps"] * (case["batch"] * 152 + npar * 28)
    return {"bytes": by, "flops": case["steps"] * case["batch"] * 8 * npar}


# ---------------------------------------------------------------------------------------
# exact: the same method in 64 bits (exact sums, each format's one rounding)
# ---------------------------------------------------------------------------------------

def _pow2(e):
    """2^e of an integer tensor, from the bit pattern (normal range)."""
    return ((e.to(torch.int64) + 1023) << 52).view(torch.float64)


def _round(x, f):
    """fl_f(x), ties to even, gradual underflow, overflow to infinity."""
    if f == F["fp64"]:
        return x
    T, emin, emax = PARAM[{5: 1, 6: 0}.get(f, f)]
    e = torch.frexp(x)[1].to(torch.int64) - 1
    quantum = _pow2(e.clamp(min=emin) - (T - 1))
    y = torch.round(x / quantum) * quantum
    big = (2.0 - 2.0 ** (1 - T)) * 2.0 ** emax
    return torch.where(y.abs() > big, torch.sign(x) * math.inf, y)


def _values(A, f):
    """The stored values in format f (as fp64), and the row scales of the row-scaled formats."""
    n, rp, _, val = A
    if f not in (F["bf16r"], F["fp16r"]):
        return _round(val, f), None
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).to(torch.int64))
    top = torch.zeros(n, dtype=torch.float64, device=DEV).scatter_reduce(0, row, val.abs(), "amax")
    s = _pow2(torch.frexp(top)[1] - 1)
    return _round(val / s[row], f), s


def _product(A, f, p, cache):
    if f not in cache:
        cache[f] = _values(A, f)
    v, s = cache[f]
    q = _round(_matvec(A, v, _round(p, f)), f)
    return q if s is None else q * s


def _diag_inverse(A):
    n, rp, ci, val = A
    row = torch.repeat_interleave(torch.arange(n, device=DEV), (rp[1:] - rp[:-1]).to(torch.int64))
    d = torch.empty(n, dtype=torch.float64, device=DEV)
    on = ci.to(torch.int64) == row
    d[row[on]] = val[on]
    return 1.0 / d


def _cg(A, b, formats, precond, iters, min_k=10, step=None):
    """The CG of the library with the formats of formats(k, rho); step(k, rho, rho_next or None)
    is told of every iteration. Returns x, iterations, outcome, actions (op, format) counts."""
    minv = _diag_inverse(A) if precond else None
    cache, counts = {}, np.zeros((4, 8), dtype=np.int64)
    dot = lambda u, v, f: float(_round((_round(u, f) * _round(v, f)).sum().reshape(1), f)[0])
    x, r = torch.zeros_like(b), b.clone()
    p = r * minv if precond else r.clone()
    sigma, bn, rho = float((r * p).sum()), float(b.norm()), 1.0
    for k in range(iters):
        f = formats(k, rho)
        for op in range(4):
            counts[op, f[op]] += 1
        q = _product(A, f[0], p, cache)
        nu = dot(p, q, f[2])
        if not (nu > 0.0) or not math.isfinite(nu) or not math.isfinite(sigma / nu):
            if step:
                step(k, rho, None, False)
            return x, k, 2, counts
        alpha = sigma / nu
        r = r - alpha * q
        x = x + alpha * p
        new = float(r.norm()) / bn
        if new < TOL and k >= min_k:
            if step:
                step(k, rho, new, True)
            return x, k + 1, 0, counts
        z = _round(r * minv if precond else r, f[1])
        snew = dot(r, z, f[3])
        if step:
            step(k, rho, new, False)
        p = z + (snew / sigma) * p
        sigma, rho = snew, new
    return x, iters, 1, counts


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x64-10 on Python integers: the first two output words."""
    mask = (1 << 64) - 1
    c = [c0, c1, c2, c3]
    for _ in range(10):
        a, b = 0xD2E7470EE14C6C93 * c[0], 0xCA5A826395121157 * c[2]
        c = [(b >> 64) ^ c[1] ^ k0, b & mask, (a >> 64) ^ c[3] ^ k1, a & mask]
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & mask, (k1 + 0xBB67AE8584CAA73B) & mask
    return c[0], c[1]


def _exact_train(case, seed):
    sysm = _train_systems(case, seed)
    cost, E = (0.8, 0.6, 0.8, 1.0, 2.0), case["episodes"]
    Q, visits = np.zeros((4, 100, 5)), np.zeros((4, 100), dtype=np.int32)
    its = np.zeros((E, len(sysm)), dtype=np.int32)

    def update(T, s, act, R, s2):
        for j in range(4):
            target = R if s2 is None else R + 0.9 * T[j, s2].max()
            T[j, s, act[j]] += 0.1 * (target - T[j, s, act[j]])

    for e in range(1, E + 1):
        eps, rounds = max(0.1, 1.0 - e / E), []
        for lane, (A, b) in enumerate(sysm):
            mine, now = Q.copy(), {}

            def formats(k, rho):
                act = [int(mine[j, _state(k, rho)].argmax()) for j in range(4)]
                for j in range(4):
                    w0, w1 = _philox(e, lane, k, j, int(seed) % 1000, 0x6D706367)
                    if (w0 >> 11) * 2.0 ** -53 < eps:
                        act[j] = (w1 & 0xFFFFFFFF) % 5
                now["act"] = act
                return act

            def step(k, rho, new, done):
                act = now["act"]
                R = (-16.0 if new is None else min(-math.log10(new), 16.0)) - 0.1 * sum(cost[a] for a in act)
                R += 10.0 if new is not None and new < TOL else 0.0
                t = (_state(k, rho), act, R, None if new is None or done else _state(k + 1, new))
                update(mine, *t)
                rounds.append(t)

            its[e - 1, lane] = _cg(A, b, formats, 0, case["iters"], step=step)[1]
        for t in rounds:
            update(Q, *t)
            for j in range(4):
                visits[j, t[0]] += 1
    return {"Q": Q, "visits": visits, "iters": its}


def _exact_mlp(case, seed):
    d, w = _transitions(case, seed)
    H, gamma, B = case["hidden"], 0.9, case["batch"]
    shapes = [(H, 16), (H,), (H, H), (H,), (20, H), (20,)]

    def split(v):
        return [t.reshape(s) for t, s in zip(torch.split(v, [int(np.prod(s)) for s in shapes]), shapes)]

    def net(v, f):
        W1, b1, W2, b2, W3, b3 = split(v)
        return (torch.relu(torch.relu(f @ W1.T + b1) @ W2.T + b2) @ W3.T + b3).reshape(-1, 4, 5)

    t64 = lambda a: torch.as_tensor(a.astype(np.float64)).to(DEV)
    f, fn, rew, done = (t64(d[k]) for k in ("f", "f_next", "reward", "done"))
    act = torch.as_tensor(d["act"].astype(np.int64)).to(DEV)
    p = t64(w)
    target, m, v = p.clone(), torch.zeros_like(p), torch.zeros_like(p)
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))  # the constants as fp32 holds them
    losses = []
    for t in range(1, case["steps"] + 1):
        idx = torch.tensor([_philox(t, b, 0, 0, 3, 0x6D6C7030)[0] % case["count"] for b in range(B)], device=DEV)
        y = rew[idx, None] + gamma * (1.0 - done[idx, None]) * net(target, fn[idx]).amax(2)
        q = p.clone().requires_grad_(True)
        out = net(q, f[idx]).gather(2, act[idx][:, :, None])[:, :, 0]
        loss = 0.5 * (out - y).square().sum() / (4 * B)
        g, = torch.autograd.grad(loss, q)
        losses.append(float(loss.detach()))
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        p = p - float(np.float32(1e-3)) * (m / (1 - b1 ** t)) / (torch.sqrt(v / (1 - b2 ** t)) + 1e-8)
        if t % 20 == 0:
            target = p.clone()
    return {"params": p.cpu().numpy(), "loss": np.array(losses)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        A, b = _system(case["family"], case["m"], seed)
        if case["precond"] == 2:
            return None  # the incomplete factor is sequential: minutes in plain torch
        x, its, outcome, counts = _cg(A, b, _formats(case["policy"]), case["precond"], case["iters"])
        x = x.cpu().numpy() if case["host"] else x
        return {"x": x, "iters": its, "outcome": outcome, "actions": counts}
    if kind == "spmv":
        m = _graph_nodes(case) if case["family"] == "graph" else case["m"]
        A, b = _system(case["family"], m, seed)
        return [_product(A, F[t], b, {}) for t in case["formats"].split(",")]
    if kind == "batch":
        got = [_cg(A, b, _formats(case["policy"]), 1, cap) for A, b, cap in _batch_systems(case, seed)]
        return {"x": torch.cat([g[0] for g in got]), "iters": np.array([g[1] for g in got])}
    if kind == "ic_batch":
        return None  # as the single solve with IC(0)
    return _exact_train(case, seed) if kind == "train" else _exact_mlp(case, seed)
