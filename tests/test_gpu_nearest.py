"""The k nearest neighbours at the edges of their forms: lists kept by the lanes (k up to 8), by the
warp in one to eight registers (32, 64, 128 and 256), with keys inserted or merged."""
import numpy as np
import pytest

import oracle

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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 31, 32, 33, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("order", ["random", "rising", "falling", "equal"])
def test_nearest_at_the_edges(aps, k, order):
    """Rows of 0 to 301 neighbours whose weights come in any order, rise, fall or tie."""
    n = 302
    i = np.concatenate([np.full(n - 1 - a, a, np.int32) for a in range(0, n, 7)])
    j = np.concatenate([np.arange(a + 1, n, dtype=np.int32) for a in range(0, n, 7)])
    s = np.random.default_rng(k).random(i.size).astype(np.float32) - np.float32(0.25)
    if order != "random":
        s = {"rising": j, "falling": -j, "equal": 0 * j}[order].astype(np.float32)
    n += 40  # and forty vertices without any
    g = aps.aps_graph_csr(i, j, s, n=n)
    try:
        nbr, w = aps.aps_graph_knn(g, k)
    finally:
        aps.aps_graph_free(g)
    rp, col, ww = oracle.graph_csr(i, j, s, n)
    onbr, ow = oracle.graph_knn(rp, col, ww, k)
    assert np.array_equal(nbr, onbr)
    assert np.array_equal(w, ow)
