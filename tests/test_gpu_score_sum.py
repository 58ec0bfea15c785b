"""How scores are summed: all of a score, prefix products included, in units of 2^-30 and rounded to
float32 once. The weights here are multiples of 2^-13 (2^-15 for long rows) whose products are exact in
float32 and multiples of that unit, so every sum is exact and every score is the float64 one, rounded;
in float32 the partial sums would need 26 bits (30) and be rounded on the way."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def aps():
    import torch

    import paper_1402_3010_gb300 as aps
    from paper_1402_3010_gb300 import _build

    _build.build()
    aps.load()
    torch.cuda.init()
    return aps


def _grid_rows(n, m, lo, hi, bits, seed):
    """Unit rows of lo to hi components on the grid of 2^-bits, products below 2^24 units; every second
    row is the one before it with other weights."""
    rng = np.random.default_rng(seed)
    idx, val, ptr = [], [], [0]
    for x in range(n):
        if x % 2 == 0:
            ids = np.sort(rng.choice(m, rng.integers(lo, hi + 1), replace=False))
        w = rng.uniform(0.8, 1.2, ids.size)
        k = np.rint(w / np.sqrt((w * w).sum()) * 2.0 ** bits)
        assert k.max() <= 4096
        idx.append(ids)
        val.append(k / 2.0 ** bits)
        ptr.append(ptr[-1] + ids.size)
    c = synth.SparseCSR(np.array(ptr, np.int64), np.concatenate(idx).astype(np.int32),
                        np.concatenate(val).astype(np.float32), n, m)
    norm = np.sqrt(np.add.reduceat(c.val.astype(np.float64) ** 2, c.indptr[:-1]))
    assert np.abs(norm - 1).max() < 1e-3
    return c


def _take(aps, p):
    try:
        return aps.pairs_to_numpy(p)
    finally:
        aps.aps_pairs_free(p)


def _dense(c):
    X = np.zeros((c.n, c.m))
    X[np.repeat(np.arange(c.n), np.diff(c.indptr)), c.idx] = c.val
    return X


# prefixes of up to 16 components (a lane each) and longer ones (a warp); x's row in shared memory and not
@pytest.mark.parametrize("lo,hi,bits,t", [(8, 30, 13, 0.3), (20, 60, 13, 0.6), (110, 140, 15, 0.5), (150, 250, 15, 0.8)])
def test_scores_are_the_exact_sums_rounded_once(aps, lo, hi, bits, t):
    c, t = _grid_rows(2400, 500, lo, hi, bits, lo), float(np.float32(t))
    h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, t)
    try:
        i, j, s = _take(aps, aps.aps_all_pairs(h))
        assert aps.aps_index_stats(h)["verified"] > 100
    finally:
        aps.aps_index_free(h)
    X = _dense(c)
    exact = (X @ X.T)  # (sums of at most 30 bits: exact in float64 in any order)
    want = np.argwhere(np.triu(exact >= t, 1))
    assert np.array_equal(np.stack([i, j], 1), want) and len(i) > 1000
    assert np.array_equal(s, exact[i, j].astype(np.float32))


def test_query_scores_are_the_exact_sums_rounded_once(aps):
    c, q, t = _grid_rows(3000, 500, 20, 60, 13, 7), _grid_rows(200, 500, 20, 60, 13, 7), float(np.float32(0.4))
    h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, t, aps.QUERYABLE)
    try:
        i, j, s = _take(aps, aps.aps_query(h, q.indptr, q.idx, q.val, q.n, t))
    finally:
        aps.aps_index_free(h)
    exact = _dense(q) @ _dense(c).T
    assert np.array_equal(np.stack([i, j], 1), np.argwhere(exact >= t)) and len(i) > 200
    assert np.array_equal(s, exact[i, j].astype(np.float32))
