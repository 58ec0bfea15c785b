"""Joins without the upper bounds (a kernel instance of their own, where every candidate's prefix is
looked up): rows around the size that is held in shared memory, prefixes short and long, many
candidates a window, alternating on one index with the joins that have the bounds."""
import numpy as np
import pytest

import oracle
import synth
from parity import compare

pytestmark = pytest.mark.gpu

NO_PARTIAL, NO_MINSIZE, NO_REMSCORE, NO_UPPER = 0x08, 0x10, 0x20, 0x40


@pytest.fixture(scope="module")
def aps():
    import torch

    import paper_1402_3010_gb300 as aps
    from paper_1402_3010_gb300 import _build

    _build.build()
    aps.load()
    torch.cuda.init()
    return aps


@pytest.mark.parametrize("build", [0, NO_UPPER, NO_MINSIZE | NO_REMSCORE | NO_UPPER, NO_PARTIAL | NO_UPPER])
@pytest.mark.parametrize("lengths", [(1, 13), (30, 35), (62, 67), (150, 300), (3, 260)])
def test_joins_with_and_without_upper_bounds(aps, lengths, build):
    n, t = 2500, float(np.float32(0.45))
    rng = np.random.default_rng([131, *lengths])
    m = 60 if lengths[1] < 20 else 700
    c = synth.sparse_vectors(n, m, rng.integers(*lengths, n), 1.0, "lognormal", 131, rng=rng)
    ref = oracle.bruteforce(c, t)
    h = aps.aps_build_index(c.indptr, c.idx, c.val, n, m, t, build)
    try:
        for flags in (NO_UPPER, 0, NO_UPPER, NO_MINSIZE | NO_UPPER, 0):  # (from the second on by the graph)
            p = aps.aps_all_pairs(h, flags)
            try:
                got = aps.pairs_to_numpy(p)
            finally:
                aps.aps_pairs_free(p)
            assert compare(*got, ref, t, n, csr=c)["pairs"] > 100
    finally:
        aps.aps_index_free(h)
