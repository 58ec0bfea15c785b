"""Results copied out of host memory and queries copied in. A result: below and above the size from
which the arrays are copied side by side, with an array left out, equal to the same result copied
from the device. Queries: as one buffer and as three, equal to the same queries on the device."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [1, 2, 40, 725, 900])  # 725 equal rows: 262,450 pairs, just above 2^18
def test_host_results_copy_whole(aps, n):
    csr = (np.arange(n + 1, dtype=np.int64), np.zeros(n, np.int32), np.ones(n, np.float32))
    got = []
    h = aps.aps_build_index(*csr, n, 1, 0.5)
    for flags in (0, aps.HOST_OUTPUT):
        p = aps.aps_all_pairs(h, flags)
        try:
            assert p.count == n * (n - 1) // 2
            got.append(aps.pairs_to_numpy(p))
            only = np.empty(p.count, np.int32)
            aps.aps_pairs_copy_to(p, None, only, None)
            assert np.array_equal(only, got[-1][1])
        finally:
            aps.aps_pairs_free(p)
    aps.aps_index_free(h)
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    k = np.arange(n)
    assert np.array_equal(got[0][0], np.repeat(k, n - 1 - k)) and np.all(got[0][2] == 1.0)


@pytest.mark.parametrize("nnz", [0, 1, 3994, 3995, 3996, 9000])  # 100 queries: 32 KB in all up to 3995 components
def test_host_queries_answer_as_device_queries(aps, nnz):
    import torch

    rng = np.random.default_rng(nnz)

    def csr(lengths, m):
        ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
        idx = np.concatenate([np.sort(rng.choice(m, k, replace=False)) for k in lengths]).astype(np.int32)
        val = rng.random(ptr[-1]) + 0.05
        row = np.repeat(np.arange(len(lengths)), lengths)
        nrm = np.sqrt(np.bincount(row, val * val, len(lengths)))
        return ptr, idx, (val / nrm[row]).astype(np.float32)

    m, nq = 200, 100
    h = aps.aps_build_index(*csr(np.full(3000, 40), m), 3000, m, 0.1, aps.QUERYABLE)
    q = csr(np.diff(np.linspace(0, nnz, nq + 1).astype(int)), m)
    got = []
    for args in (q, tuple(torch.from_numpy(a).cuda() for a in q)):
        p = aps.aps_query(h, *args, nq, 0.2)
        try:
            got.append(aps.pairs_to_numpy(p))
        finally:
            aps.aps_pairs_free(p)
    aps.aps_index_free(h)
    assert nnz < 100 or got[0][0].size > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)
