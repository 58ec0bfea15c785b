"""The sorts of 32-bit keys with a payload (dimension ranks, posting lists, the join's work list) at the
edges of their forms: up to 8192 items one launch, up to 1024 an SM tiles of 1024 items, above that
tiles of 5120. One index of as many one-component rows and dimensions as there are items runs all three."""
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


def _sizes():
    small = [2, 31, 33, 1023, 1025, 8191, 8192, 8193, 9216, 9217]
    return small + [f"sms{d:+d}" for d in (-1, 0, 1)] + [f"tiles{d:+d}" for d in (-1, 0, 1)] + [1000003]


@pytest.mark.parametrize("few", [False, True])  # most dimensions hold one row; 50 each
@pytest.mark.parametrize("size", _sizes())
def test_index_sorts_at_the_edges_of_their_forms(aps, size, few):
    import torch

    if isinstance(size, str):  # 1024 items an SM; whole tiles of 5120 above that
        most = torch.cuda.get_device_properties(0).multi_processor_count * 1024
        n = (most if size.startswith("sms") else (most // 5120 + 2) * 5120) + int(size[-2:])
    else:
        n = size
    rng = np.random.default_rng([121, n, few])
    # (few: 50 rows a dimension, so that ties and runs of equal keys are long)
    dim = rng.integers(0, max(n // 50, 1) if few else n, n).astype(np.int32)
    h = aps.aps_build_index(np.arange(n + 1, dtype=np.int64), dim, np.ones(n, np.float32), n, n, 0.9)
    try:
        ex = aps.aps_index_export(h)
        p = aps.aps_all_pairs(h)
        count = int(p.count)
        aps.aps_pairs_free(p)
    finally:
        aps.aps_index_free(h)
    nnz_d = np.bincount(dim, minlength=n)
    order = np.argsort(-nnz_d, kind="stable")  # decreasing count, ties by id
    rank = np.empty(n, np.int64)
    rank[order] = np.arange(n)
    assert np.array_equal(ex["rank_of_dim"], rank)
    assert np.array_equal(ex["list_ptr"], np.concatenate([[0], np.cumsum(nnz_d[order])]))
    assert np.array_equal(ex["post_id"], np.argsort(rank[dim], kind="stable"))
    assert count == int((nnz_d * (nnz_d - 1) // 2).sum())
