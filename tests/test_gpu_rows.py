"""What the index build decides about a row in float32 where that is clear and in float64 where it
is not: its norm, and where the sum of its values times the dimensions' maxima reaches t. Rows of
one and of many chunks of 32, sums that meet t exactly, thresholds whose products underflow."""
from fractions import Fraction

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


def rows(lengths, m, equal, seed):
    rng = np.random.default_rng(seed)
    ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    idx = np.concatenate([np.sort(rng.choice(m, k, replace=False)) for k in lengths]).astype(np.int32)
    val = np.ones(ptr[-1]) if equal else rng.random(ptr[-1]) + 0.01
    nrm = np.sqrt(np.add.reduceat(val * val, ptr[:-1]))
    return ptr, idx, (val / np.repeat(nrm, lengths)).astype(np.float32)


@pytest.mark.parametrize("t", [1.0, 0.75, 0.5, 0.0625, 1e-20, 1e-36])
@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("lengths", [[4, 16, 64, 1, 2, 31, 32, 33] * 20, [4096, 1024, 2047, 2048, 2049, 2500] * 4])
def test_split_is_the_float64_one(aps, t, equal, lengths):
    m = 300 if max(lengths) < 100 else 6000
    ptr, idx, val = rows(lengths, m, equal, seed=len(lengths))
    t = np.float32(t)
    h = aps.aps_build_index(ptr, idx, val, len(lengths), m, float(t))
    try:
        ex = aps.aps_index_export(h)
    finally:
        aps.aps_index_free(h)
    mwr = np.empty(m, np.float32)
    mwr[ex["rank_of_dim"]] = ex["mw_d"]
    for x in range(len(lengths)):
        a, b = ptr[x], ptr[x + 1]
        total, want = Fraction(0), {int(b - a)}
        for p in range(a, b):
            total += Fraction(float(ex["cval"][p])) * Fraction(float(mwr[ex["crank"][p]]))
            if abs(float(total) - float(t)) < 1e-12 * float(t):
                want.add(int(p - a))  # (next to t the float64 sum's own rounding decides)
            elif total >= Fraction(float(t)):
                want = want - {int(b - a)} | {int(p - a)}
                break
        assert int(ex["split"][x]) in want, (x, lengths[x])


@pytest.mark.parametrize("length", [1, 7, 300, 8192, 9000])
@pytest.mark.parametrize("norm,subunit,ok", [(1.0, False, True), (1.00099, False, True), (0.99901, False, True),
                                             (1.00101, False, False), (0.99899, False, False), (0.5, True, True),
                                             (1.00099, True, True), (1.00101, True, False), (0.5, False, False)])
def test_norms_at_the_tolerance(aps, length, norm, subunit, ok):
    ptr, idx, val = rows([length] * 3, 10000, False, seed=length)
    val[ptr[1]:ptr[2]] *= np.float32(norm)
    flags = aps.SUBUNIT_NORMS if subunit else 0
    if ok:
        aps.aps_index_free(aps.aps_build_index(ptr, idx, val, 3, 10000, 0.5, flags))
    else:
        with pytest.raises(aps.APSError):
            aps.aps_build_index(ptr, idx, val, 3, 10000, 0.5, flags)
