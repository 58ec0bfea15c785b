"""A result copied out of host memory: below and above the size from which the arrays are copied
side by side, with an array left out, and equal to the same result copied from the device."""
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
