"""Indexes whose table of window starts would outgrow the rest of the index: short lists have the
starts of groups of windows only and the join searches the lists in between. Memory in proportion to
the index, and every form of the join against the oracle."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import synth
from parity import compare

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WINDOW = 1792  # ids of a window (G = 2, 4 and 8)


@pytest.fixture(scope="module")
def aps():
    import torch

    import paper_1402_3010_gb300 as aps
    from paper_1402_3010_gb300 import _build

    _build.build()
    aps.load()
    torch.cuda.init()
    return aps


def _set(n, m, seed, longest=200):
    """Rows of one to four components, some of up to `longest`, every tenth the row before it with other
    weights; far more dimensions than the rows can fill."""
    rng = np.random.default_rng([105, seed])
    lengths = rng.integers(1, 5, n)
    lengths[::23] = rng.integers(20, longest, lengths[::23].size)
    lengths[9::10] = lengths[8::10][:lengths[9::10].size]
    c = synth.sparse_vectors(n, m, lengths, 0.6, "uniform", 105, rng=rng)
    for x in range(9, n, 10):
        a, b, z = int(c.indptr[x - 1]), int(c.indptr[x]), int(c.indptr[x + 1])
        if z - b != b - a:
            continue
        v = c.val[a:b].astype(np.float64) * rng.uniform(1.0, 1.3, b - a)
        c.idx[b:z] = c.idx[a:b]
        c.val[b:z] = (v / np.sqrt((v * v).sum())).astype(np.float32)
    return c


def _past_its_share(c):
    """Whether the table with every window takes more than 32 bytes a component and 16 a dimension."""
    return 4 * c.m * (-(-c.n // WINDOW) + 1) > 32 * c.nnz + 16 * c.m


def _take(aps, p):
    try:
        return aps.pairs_to_numpy(p)
    finally:
        aps.aps_pairs_free(p)


# windows, and how many a group holds: 12 in twos, 12 in fours, 16 in eights, 4 in twos
@pytest.mark.parametrize("n,m", [(21000, 200000), (21000, 800000), (27000, 1200000), (5400, 400000)])
def test_joins_with_groups_of_windows_match_the_oracle(aps, n, m):
    import torch

    t = float(np.float32(0.6))
    c = _set(n, m, n)
    assert _past_its_share(c)
    ref = oracle.bruteforce(c, t)
    h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, t)
    try:
        first = _take(aps, aps.aps_all_pairs(h))
        r = compare(*first, ref, t, n, csr=c)
        assert r["pairs"] > n // 10
        for flags in (0, 0x10, 0x20, 0x40):  # again (the graph), without minsize, remscore, upperbound
            got = _take(aps, aps.aps_all_pairs(h, flags))
            assert np.array_equal(got[0], first[0]) and np.array_equal(got[1], first[1])
        for nblk, heavy in ((2, 300), (4, n)):
            compare(*_take(aps, aps.aps_all_pairs_split(h, nblk, heavy)), ref, t, n, csr=c)
        k = len(first[0])
        out = [torch.empty(k + 8, dtype=d, device="cuda") for d in (torch.int32, torch.int32, torch.float32)]
        assert aps.aps_all_pairs_noalloc(h, *out) == k
        for a, b in zip(out, first):
            assert np.array_equal(a[:k].cpu().numpy(), b)
    finally:
        aps.aps_index_free(h)


@pytest.mark.parametrize("n,m", [(21000, 800000), (27000, 1200000)])
def test_queries_with_groups_of_windows_match_the_oracle(aps, n, m):
    t = float(np.float32(0.6))
    c = _set(n, m, n + 1)
    assert _past_its_share(c)
    step = n // 400
    at = np.concatenate([np.arange(c.indptr[x], c.indptr[x + 1]) for x in range(0, n, step)])
    rows = np.arange(0, n, step)
    ptr = np.concatenate([[0], np.cumsum(np.diff(c.indptr)[rows])]).astype(np.int64)
    q = synth.SparseCSR(ptr, c.idx[at], c.val[at], len(rows), m)
    ref = oracle.bruteforce_cross(q, c, t)
    h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, t, aps.QUERYABLE)
    try:
        got = _take(aps, aps.aps_query(h, q.indptr, q.idx, q.val, q.n, t))
    finally:
        aps.aps_index_free(h)
    assert compare(*got, ref, t, n, self_join=False, csr=c, queries=q)["pairs"] >= len(rows)


def test_batch_with_groups_of_windows_matches_the_oracle(aps):
    """One instance sets how coarse the table is; the others have fewer windows than a group holds."""
    t = float(np.float32(0.6))
    sets = [_set(26000, 900000, 1), _set(5000, 3000, 2, longest=40), _set(40, 2000, 3), _set(9000, 90000, 4)]
    assert _past_its_share(sets[0])
    outs, _ = aps.aps_batch_all_pairs([(c.indptr, c.idx, c.val, c.n, c.m, t) for c in sets])
    for p, c in zip(outs, sets):
        compare(*_take(aps, p), oracle.bruteforce(c, t), t, c.n, csr=c)


def test_many_windows_and_clustered_lists(aps):
    """67 windows: lists of up to 8 entries are coarser, in groups of 2 to 16 windows. Blocks of 30
    neighbouring rows share dimensions of their own, so some groups hold a whole list."""
    t, n, m = float(np.float32(0.8)), 120000, 1000000
    rng = np.random.default_rng(106)
    lengths = rng.integers(1, 4, n)
    c = synth.sparse_vectors(n, m - 30000, lengths, 0.2, "uniform", 106, rng=rng)
    idx, val, ptr = [], [], [0]
    for x in range(n):
        i, v = c.row(x)
        if x % 300 < 30:  # a block: two dimensions of its own, in most of its rows
            own = m - 30000 + 2 * (x // 300)
            take = [own, own + 1] if x % 7 else [own]
            i, v = np.concatenate([i[:1], take]), np.concatenate([v[:1] * 0.2, rng.random(len(take)) + 0.5])
        idx.append(i)
        val.append(v / np.sqrt(np.sum(v.astype(np.float64) ** 2)))
        ptr.append(ptr[-1] + len(i))
    c = synth.SparseCSR(np.array(ptr, np.int64), np.concatenate(idx).astype(np.int32),
                        np.concatenate(val).astype(np.float32), n, m)
    assert _past_its_share(c)
    h = aps.aps_build_index(c.indptr, c.idx, c.val, n, m, t)
    try:
        got = _take(aps, aps.aps_all_pairs(h))
        split = _take(aps, aps.aps_all_pairs_split(h, 2, 5000))
    finally:
        aps.aps_index_free(h)
    ref, _ = oracle.all_pairs(c, t)
    assert compare(*got, ref, t, n, csr=c)["pairs"] > 20000
    compare(*split, ref, t, n, csr=c)


SIZE = """
import numpy as np, torch
import paper_1402_3010_gb300 as aps
n, m = 300000, 2000000
rng = np.random.default_rng(1)
idx = np.sort(rng.integers(0, m // 10, (n, 10)) * 10 + np.arange(10), axis=1).astype(np.int32)
val = np.full((n, 10), 10 ** -0.5, np.float32)
dev = [torch.from_numpy(a).cuda() for a in (np.arange(n + 1, dtype=np.int64) * 10, idx.ravel(), val.ravel())]
aps.aps_index_free(aps.aps_build_index(np.zeros(2, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32), 1, 1, 0.9))
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
h = aps.aps_build_index(*dev, n, m, 0.9)
print(before - torch.cuda.mem_get_info()[0])
"""


def test_wide_sparse_index_takes_memory_in_proportion(aps):
    """300,000 rows of ten components over two million dimensions: the table with every window would be
    1.35 GB. 3M components and 2M dimensions: at most 128 MB for the table; the build's other arrays and
    scratch are at most 100 bytes a component, 64 a dimension and 200 a row, 490 MB."""
    r = subprocess.run([sys.executable, "-c", SIZE], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    assert int(r.stdout) < 128e6 + 490e6, int(r.stdout)
