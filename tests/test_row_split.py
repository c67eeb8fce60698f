"""Row split of CSR operators over the CTAs (host): every row once, in order, at most
`cap` rows per CTA, and every boundary within half a row of its place, for
even, empty and very uneven rows and for more CTAs than rows."""

import numpy as np
import pytest

from paper_1102_5071_gb300 import _capi
from paper_1102_5071_gb300.build import build

ROW_COST = 8  # entries that the vector passes over one row count as


@pytest.fixture(scope="module")
def lib():
    build()
    return _capi.load()


def _counts(kind, nops, dim, rng):
    if kind == "even":
        return np.full((nops, dim), 5)
    if kind == "empty":
        return np.zeros((nops, dim), dtype=int)
    if kind == "one-long":
        c = np.zeros((nops, dim), dtype=int)
        c[0, dim // 2] = 100000
        return c
    if kind == "head":  # all the work in the first rows
        c = np.ones((nops, dim), dtype=int)
        c[:, : max(1, dim // 50)] = 900
        return c
    return (rng.pareto(1.0, (nops, dim)) * 10).astype(int).clip(0, 5000)


@pytest.mark.parametrize("kind", ["even", "empty", "one-long", "head", "pareto"])
@pytest.mark.parametrize("dim,grid", [(1, 1), (1, 7), (3, 152), (152, 152), (153, 152), (1000, 3), (20011, 152)])
@pytest.mark.parametrize("tight", [False, True])
def test_row_split(lib, kind, dim, grid, tight):
    nops = 2
    n = _counts(kind, nops, dim, np.random.default_rng(dim + grid))
    rp, base = [], 0
    for o in range(nops):
        rp.append(base + np.concatenate(([0], np.cumsum(n[o]))))
        base = int(rp[-1][-1])
    rp = np.ascontiguousarray(np.concatenate(rp), dtype=np.int32)
    cap = -(-dim // grid) if tight else 1 << 30  # tight: every CTA has to take all it may
    rb = np.full(grid + 1, -1, dtype=np.int32)
    assert lib.cfet_selftest_row_split(rp.ctypes.data, nops, dim, grid, cap, rb.ctypes.data) == _capi.CFET_OK
    assert rb[0] == 0 and rb[grid] == dim
    rows = np.diff(rb)
    assert (rows >= 0).all() and (rows <= cap).all()
    if not tight:
        work = n.sum(axis=0) + ROW_COST
        cum = np.concatenate(([0], np.cumsum(work)))
        mean = cum[-1] / grid
        for b in range(grid):
            mine = work[rb[b]: rb[b + 1]]
            # a boundary is off its place by half a row at most on either side
            assert mine.sum() <= mean + 2 + (mine[0] / 2 + mine[-1] / 2 if len(mine) else 0)
