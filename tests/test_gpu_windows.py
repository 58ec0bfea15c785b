"""GPU parity of the join's windows: set sizes at the edges of a window, windows whose candidates
overrun a warp's list, rows around the sizes that stay in registers and in shared memory, runs
that go over several staging slabs, and two-component rows whose lists are too long to stream."""
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


def _check(aps, c, t, flags=0):
    t = float(np.float32(t))
    h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, t, flags)
    try:
        p = aps.aps_all_pairs(h)
        try:
            got = aps.pairs_to_numpy(p)
        finally:
            aps.aps_pairs_free(p)
    finally:
        aps.aps_index_free(h)
    return compare(*got, oracle.bruteforce(c, t), t, c.n, csr=c)


@pytest.mark.parametrize("flags", [0, 0x40, 0x20])  # every bound; no prefix bound; no remscore
@pytest.mark.parametrize("n", [2, 1791, 1792, 1793, 3585])
def test_dense_windows_overrun_the_candidate_list(aps, n, flags):
    """40 dimensions: nearly every slot of a window is a candidate, and every vector has matches."""
    rng = np.random.default_rng([91, n])
    c = synth.sparse_vectors(n, 40, rng.integers(1, 13, n), 0.8, "uniform", 91, rng=rng)
    r = _check(aps, c, 0.6, flags)
    assert n < 100 or r["pairs"] > 5 * n


@pytest.mark.parametrize("lengths", [(30, 35), (62, 67), (150, 300)])
def test_rows_around_the_register_and_shared_memory_sizes(aps, lengths):
    rng = np.random.default_rng([92, lengths[0]])
    n = 2500
    c = synth.sparse_vectors(n, 700, rng.integers(*lengths, n), 1.0, "lognormal", 92, rng=rng)
    assert _check(aps, c, 0.5)["pairs"] > 100


def test_two_component_rows_with_long_lists(aps):
    """Rows of two of three dimensions: the pairs of lists are past what one warp streams (8192
    entries), the rows go by windows, and runs of matches go over several staging slabs."""
    n = 14000
    rng = np.random.default_rng(93)
    c = synth.sparse_vectors(n, 3, np.full(n, 2), 0.3, "uniform", 93, rng=rng)
    assert _check(aps, c, 0.97)["pairs"] > 100 * n
