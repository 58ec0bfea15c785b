"""The radix sort at the edges of its forms and tiles, through the calls that sort: the graph
build (64-bit keys with a payload) and the candidate union (64-bit keys alone, with repeats).
Up to 8192 items take the one-launch form, up to 1024 for each of 152 SMs tiles of 1024, more the
form of 4096-item tiles. Both results are whole numbers and copied weights, so they are compared exactly."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

COUNTS = [1, 31, 257, 3072, 8191, 8192, 8193, 3 * 3072 - 1, 3 * 3072, 3 * 3072 + 1, 70001,
          152 * 1024, 152 * 1024 + 1, 40 * 4096 - 1, 40 * 4096, 40 * 4096 + 1]


@pytest.fixture(scope="module")
def aps():
    import torch

    import paper_1402_3010_gb300 as aps
    from paper_1402_3010_gb300 import _build

    _build.build()
    aps.load()
    torch.cuda.init()
    return aps


def pairs(n, count, seed):
    """count distinct pairs i < j of [0, n) in (i, j) order."""
    rng = np.random.default_rng(seed)
    key = np.zeros(0, np.int64)
    while key.size < count:
        a, b = rng.integers(0, n, count + 100), rng.integers(0, n, count + 100)
        ok = a != b
        key = np.unique(np.concatenate([key, np.minimum(a, b)[ok] * n + np.maximum(a, b)[ok]]))
    key = np.sort(rng.choice(key, count, replace=False))
    return (key // n).astype(np.int32), (key % n).astype(np.int32), rng.random(count).astype(np.float32)


@pytest.mark.parametrize("n", [1000, 70000, 20_000_000])
@pytest.mark.parametrize("count", COUNTS)
def test_pairs_with_a_payload(aps, n, count):
    i, j, s = pairs(n, count, seed=count + n)
    g = aps.aps_graph_csr(i, j, s, n=n)
    try:
        got = aps.graph_to_numpy(g)
    finally:
        aps.aps_graph_free(g)
    for a, b in zip(got, oracle.graph_csr(i, j, s, n)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("count", COUNTS)
def test_keys_alone_with_repeats(aps, count):
    n = 5000
    i, j, _ = pairs(n, count, seed=count)
    pick = np.random.default_rng(count).integers(0, count, count)  # any order, some twice
    lists, held = [], []
    for part in np.array_split(pick, 2):
        a, b = np.ascontiguousarray(i[part]), np.ascontiguousarray(j[part])
        lists.append(aps.aps_pairs(count=part.size, i=a.ctypes.data, j=b.ctypes.data))
        held += [a, b]
    # one dimension, every row 1 in it: each pair of the union scores 1
    out, nc = aps.aps_pairs_verify(lists, np.arange(n + 1, dtype=np.int64), np.zeros(n, np.int32),
                                   np.ones(n, np.float32), n, 1, 0.5)
    try:
        gi, gj, gs = aps.pairs_to_numpy(out)
    finally:
        aps.aps_pairs_free(out)
    want = np.unique(pick)  # positions in (i, j) order
    assert nc == want.size
    assert np.array_equal(gi, i[want]) and np.array_equal(gj, j[want]) and np.all(gs == 1.0)
