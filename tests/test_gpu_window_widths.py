"""Sets of few vectors are joined with narrower windows (a half, a quarter or an eighth of 1792 ids, so
that a heavy vector's windows can be cut into parts): at the sizes where the width changes, for
self-joins, queries, the split and allocation-free joins, and batches of small instances."""
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


def _take(aps, p):
    try:
        return aps.pairs_to_numpy(p)
    finally:
        aps.aps_pairs_free(p)


def _set(n, seed):
    """Rows of 1 to 12 of 100 dimensions, some of 60 to 80: most slots of a window are candidates."""
    rng = np.random.default_rng([141, seed, n])
    lengths = rng.integers(1, 13, n)
    lengths[::97] = rng.integers(60, 81, lengths[::97].size)
    return synth.sparse_vectors(n, 100, lengths, 0.5, "uniform", 141, rng=rng)


@pytest.mark.parametrize("n", [3, 671, 672, 673, 1791, 1792, 3583, 3584, 7167, 7168])
def test_self_joins_at_the_sizes_where_the_width_changes(aps, n):
    import torch

    c, t = _set(n, 0), float(np.float32(0.9))
    ref = oracle.bruteforce(c, t)
    h = aps.aps_build_index(c.indptr, c.idx, c.val, n, c.m, t)
    try:
        first = _take(aps, aps.aps_all_pairs(h))
        compare(*first, ref, t, n, csr=c)
        assert len(first[0]) > n // 10 or n < 1000
        compare(*_take(aps, aps.aps_all_pairs_split(h, 3, max(n // 50, 1))), ref, t, n, csr=c)
        out = [torch.empty(len(first[0]) + 8, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.float32)]
        assert aps.aps_all_pairs_noalloc(h, *out) == len(first[0])
        for a, b in zip(out, first):
            assert np.array_equal(a[:len(b)].cpu().numpy(), b)
    finally:
        aps.aps_index_free(h)


@pytest.mark.parametrize("groups", [1, 2])  # (G = 1: windows of 4096 ids and their halves)
@pytest.mark.parametrize("n", [100, 1791, 3584, 7168, 16384])
def test_queries_and_tile_shapes(aps, n, groups):
    c, t = _set(n, 1), float(np.float32(0.85))
    q = _set(150, 2)
    before = aps.aps_get_tuning(), aps.aps_get_tuning(True)
    try:
        aps.aps_set_tuning([groups] * 8, [groups] * 8)
        h = aps.aps_build_index(c.indptr, c.idx, c.val, n, c.m, t, aps.QUERYABLE)
    finally:
        aps.aps_set_tuning(*before)
    try:
        got = _take(aps, aps.aps_query(h, q.indptr, q.idx, q.val, q.n, t))
        compare(*got, oracle.bruteforce_cross(q, c, t), t, n, self_join=False, csr=c, queries=q)
        compare(*_take(aps, aps.aps_all_pairs(h)), oracle.bruteforce(c, t), t, n, csr=c)
    finally:
        aps.aps_index_free(h)


def test_batch_of_small_instances(aps):
    t = float(np.float32(0.9))
    sets = [_set(n, 3) for n in (500, 2, 1800, 230, 1, 900)]  # 3433 rows in all
    outs, _ = aps.aps_batch_all_pairs([(c.indptr, c.idx, c.val, c.n, c.m, t) for c in sets])
    for p, c in zip(outs, sets):
        compare(*_take(aps, p), oracle.bruteforce(c, t), t, c.n, csr=c)


def test_noalloc_pairs_that_fit_the_arena_without_parts_alone(aps):
    """3745 equal rows: 7,010,640 pairs. The arena stages 7,069,248 where each vector has one slot, and
    6,938,560 with the slots of nine parts a vector: the join runs again in one part."""
    import torch

    n = 3745
    ptr = np.arange(n + 1, dtype=np.int64) * 3
    idx, val = np.tile(np.arange(3, dtype=np.int32), n), np.full(3 * n, 3 ** -0.5, np.float32)
    h = aps.aps_build_index(ptr, idx, val, n, 3, 0.9)
    try:
        want = n * (n - 1) // 2
        out = [torch.empty(want, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.float32)]
        assert aps.aps_all_pairs_noalloc(h, *out) == want
    finally:
        aps.aps_index_free(h)
    i, j = np.triu_indices(n, 1)
    assert np.array_equal(out[0].cpu().numpy(), i) and np.array_equal(out[1].cpu().numpy(), j)
    assert np.abs(out[2].cpu().numpy() - 1).max() < 1e-5
