"""The paper's upperbound (Sec. 3.2.2) does its own work: of the candidates that the norm bound lets
through, those with A[y] + min(|y'|, |x|) * maxweight(x) * maxweight(y') < t get no dot(x, y')."""
import numpy as np
import pytest

import oracle
import synth
from parity import compare

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


def _flat_rows(n, m, seed):
    """Rows of 64 equal weights (1/8, so that every sum of products is exact) and, so that prefixes are
    short, one row of four weights 1/2 for every four dimensions."""
    rng = np.random.default_rng(seed)
    rows = [np.sort(rng.choice(m, 64, replace=False)) for _ in range(n)]
    rows[1::20] = rows[0::20]
    heavy = [np.arange(d, d + 4) for d in range(0, m, 4)]
    idx = np.concatenate(rows + heavy).astype(np.int32)
    lengths = [64] * n + [4] * len(heavy)
    val = np.repeat([0.125] * n + [0.5] * len(heavy), lengths).astype(np.float32)
    return synth.SparseCSR(np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64), idx, val, n + len(heavy), m)


@pytest.mark.parametrize("variant", ["all-pairs-1-upperbound", "all-pairs-1-array", "all-pairs-2"])
def test_upperbound_prunes_what_the_norm_bound_lets_through(aps, variant):
    c, t = _flat_rows(600, 400, 111), float(np.float32(0.4))
    h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, t, aps.VARIANTS[variant])
    try:
        ex = aps.aps_index_export(h)
        p = aps.aps_all_pairs(h)
        try:
            got = aps.pairs_to_numpy(p)
        finally:
            aps.aps_pairs_free(p)
        verified = aps.aps_index_stats(h)["verified"]
    finally:
        aps.aps_index_free(h)
    compare(*got, oracle.bruteforce(c, t), t, c.n, csr=c)
    # y's prefix: up to the split and, with every bound on, to where its norm can reach t (the join's own lists)
    split = ex["split"].copy()
    if variant == "all-pairs-2":
        for x in range(c.n):
            a, b = int(c.indptr[x]), int(c.indptr[x + 1])
            reach = np.nonzero(np.cumsum(ex["cval"][a:b].astype(np.float64) ** 2) * 1.0025 >= t * t)[0]
            split[x] = max(split[x], reach[0] if reach.size else b - a)
    # the pairs that share a component of y's indexed part, by what bounds them
    X, Y, P = (np.zeros((c.n, c.m)) for _ in range(3))
    for x in range(c.n):
        a, b, sp = int(c.indptr[x]), int(c.indptr[x + 1]), int(split[x])
        X[x, ex["crank"][a:b]] = ex["cval"][a:b]
        Y[x, ex["crank"][a + sp:b]] = ex["cval"][a + sp:b]
        P[x, ex["crank"][a:a + sp]] = ex["cval"][a:a + sp]
    A = X @ Y.T
    later = (np.arange(c.n)[:, None] < np.arange(c.n)) & (A > 0) & (split > 0)
    upper = np.minimum(split, ex["len"][:, None]) * ex["mw"][:, None] * P.max(1)
    allowed = int((later & (A + upper >= t - 1e-5)).sum())
    if variant == "all-pairs-1-array":  # without the bounds every candidate with a prefix is verified
        assert verified == int(later.sum())
        return
    # the norm bound alone lets through far more: ||x on the ranks before y's first indexed one|| * ||y'||
    first = np.array([ex["crank"][c.indptr[y] + s] if s < n else c.m for y, (s, n) in enumerate(zip(split, ex["len"]))])
    norm = np.sqrt(np.cumsum(X ** 2, axis=1)[:, np.maximum(first - 1, 0)]) * np.sqrt((P ** 2).sum(1))
    assert int((later & (A + norm >= t)).sum()) > 10 * allowed
    assert verified <= allowed
