"""The ring of level blocks of the IC(0) team solver (csrc/ic_ring.h, no GPU): for the grids up to
32768 rows the places are accepted only if producer and consumers cannot end up waiting for one
another, checked by running the two against each other, and no block is overwritten before it is
consumed. The blocks' sizes are those of the packing: per level a header of 16 bytes, then per 32 rows
256 bytes and 768 per four entries of the longest row (one, two, or a multiple of four such quads)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2504_14268_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
INFLIGHT, RING, SHARED = 32, 96 * 1024, 180 * 1024

SHIM = """
#include "ic_ring.h"
extern "C" int places(mpcg::IcBlock* b, int count, int cap, int inflight) {
  std::vector<mpcg::IcBlock> v(b, b + count);
  const bool ok = mpcg::ic_ring_places(v, cap, inflight);
  std::copy(v.begin(), v.end(), b);
  return ok ? 1 : 0;
}
"""


@pytest.fixture(scope="module")
def places(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    src, lib = d / "shim.cpp", d / "shim.so"
    src.write_text(SHIM)
    inc = os.path.join(ROOT, "paper_2504_14268_gb300", "csrc")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-fPIC", "-shared", "-I" + inc, "-o", str(lib), str(src)])
    f = ctypes.CDLL(str(lib)).places

    def call(sizes, cap, inflight=INFLIGHT):
        b = np.zeros((len(sizes), 4), dtype=np.int32)
        b[:, 1] = sizes
        ok = f(b.ctypes.data_as(ctypes.c_void_p), len(sizes), int(cap), int(inflight))
        return bool(ok), b

    return call


def _stencil(shape, full):
    """Pattern of the 7- or 27-point stencil on a 3D grid: (n, row_ptr, col)."""
    n = int(np.prod(shape))
    idx = np.arange(n).reshape(shape)
    rows, cols = [], []
    for d in np.ndindex(3, 3, 3):
        o = np.array(d) - 1
        if not full and np.abs(o).sum() > 1:
            continue
        a = tuple(slice(max(0, -s), m - max(0, s)) for s, m in zip(o, shape))
        b = tuple(slice(max(0, s), m - max(0, -s)) for s, m in zip(o, shape))
        rows.append(idx[a].ravel())
        cols.append(idx[b].ravel())
    r, c = np.concatenate(rows), np.concatenate(cols)
    order = np.lexsort((c, r))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))])
    return n, rp.astype(np.int32), c[order].astype(np.int32)


def _blocks(A):
    """16-byte units of every level's block, forward then backward, and the ring that the vector leaves."""
    from paper_2504_14268_gb300 import mpcg

    n, rp, ci = A[:3]
    lo, up, depth = mpcg.csr_levels(A)
    r = np.repeat(np.arange(n), np.diff(rp))
    units = []
    for lev, d, mine in ((lo, depth[0], ci < r), (up, depth[1], ci > r)):
        length = np.bincount(r[mine], minlength=n)
        longest = np.zeros(d, dtype=int)
        np.maximum.at(longest, lev, length)
        groups = (np.bincount(lev, minlength=d) + 31) // 32
        quads = np.where(longest <= 4, 1, np.where(longest <= 8, 2, (longest + 15) // 16 * 4))
        units += list(1 + groups * (256 + 768 * quads) // 16)
    fit = SHARED - 8 * ((n + 2) // 2)
    return units, min(RING, fit, 16 * sum(units)) // 16


def _runs(b):
    """Producer against consumers: None when all levels are consumed from intact blocks, else where
    both wait (or a block is lost)."""
    issued, done, ring = 0, 0, {}
    for level in range(len(b)):  # the barrier before `level`: its block is here
        while issued <= level or (issued < len(b) and b[issued, 3] <= done):
            if b[issued, 3] > done:
                return f"block {issued} waits for level {b[issued, 3] - 1}, level {level} for block {issued}"
            lo, hi = b[issued, 2], b[issued, 2] + b[issued, 1]
            ring = {j: v for j, v in ring.items() if v[1] <= lo or hi <= v[0]}
            ring[issued] = (lo, hi)
            issued += 1
        done = level  # levels before this one are consumed
        if level not in ring:
            return f"level {level} overwritten"
    return None


GRIDS = [((m, m, m), full) for m in (28, 29, 30, 31, 32) for full in (True, False)] + [
    ((20, 40, 40), False), ((20, 40, 40), True), ((181, 181, 1), False), ((1024, 4, 8), True), ((8, 64, 64), False)]


@pytest.mark.parametrize("shape,full", GRIDS)
def test_accepted_rings_run_to_the_end(places, shape, full):
    A = _stencil(shape, full)
    assert A[0] <= 32768
    units, cap = _blocks(A)
    ok, b = places(units, cap)
    if ok:
        assert (b[:, 2] >= 0).all() and (b[:, 2] + b[:, 1] <= cap).all()
        assert _runs(b) is None
    else:  # ... and what is refused could not have run: a neighbour's place, or a block beyond the ring
        l = next(i for i in range(1, len(units)) if b[i, 3] == 0 and b[i, 2] < b[i - 1, 2] + b[i - 1, 1])
        assert b[l, 2] + b[l, 1] > b[l - 1, 2]
    if shape == (28, 28, 28):
        assert ok  # ring of the full 96 KB


def test_grids_beyond_the_ring_are_refused(places):
    """Three blocks of the widest levels exceed the ring beside the vector of these systems."""
    for shape, full in (((30, 30, 30), True), ((31, 31, 31), True), ((32, 32, 32), True), ((31, 31, 31), False),
                        ((32, 32, 32), False), ((20, 40, 40), False)):
        units, cap = _blocks(_stencil(shape, full))
        assert 3 * max(units) > cap
        assert not places(units, cap)[0], (shape, full)


def test_small_cases(places):
    assert places([5], 5)[0] and not places([6], 5)[0]
    assert places([3, 3], 6)[0] and not places([3, 3], 5)[0]
    ok, b = places([2, 2, 2, 2], 4)  # two places in turn
    assert ok and list(b[:, 2]) == [0, 2, 0, 2] and list(b[:, 3]) == [0, 0, 1, 2] and _runs(b) is None
    ok, b = places([1] * 9, 100, inflight=4)
    assert ok and list(b[:, 3]) == [0, 0, 0, 0, 1, 2, 3, 4, 5] and _runs(b) is None
    rng = np.random.default_rng(0)
    for _ in range(300):
        sizes = rng.integers(1, 12, rng.integers(1, 40))
        ok, b = places(sizes, rng.integers(12, 40), inflight=int(rng.integers(2, 9)))
        if ok:
            assert _runs(b) is None
