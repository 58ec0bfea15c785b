"""Dense rows whose norm is at the tolerance (float32 decides clear ones, float64 the rest), and the
scores of candidate lists with one and with several rows i, at every register count of a row."""
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


@pytest.mark.parametrize("d", [64, 128, 256, 320, 512])
@pytest.mark.parametrize("norm,ok", [(1.00099, True), (0.99901, True), (1.00101, False), (0.99899, False)])
def test_dense_norms_at_the_tolerance(aps, d, norm, ok):
    import torch

    x = np.random.default_rng(d).standard_normal((5, d))
    x = (x / np.linalg.norm(x, axis=1, keepdims=True)).astype(np.float32)
    x[3] = x[1]
    x[3] *= np.float32(norm)
    if not ok:
        with pytest.raises(aps.APSError):
            aps.aps_all_pairs_dense(torch.from_numpy(x).cuda(), 0.9)
        return
    p, _ = aps.aps_all_pairs_dense(torch.from_numpy(x).cuda(), 0.9)
    try:
        i, j, s = aps.pairs_to_numpy(p)
    finally:
        aps.aps_pairs_free(p)
    assert list(zip(i, j)) == [(1, 3)]
    exact = float(x[1].astype(np.float64) @ x[3].astype(np.float64))
    # (d / 32 + 5 additions in a lane and across them, each rounded to 2^-24 of the unit sum)
    assert abs(float(s[0]) - exact) <= (d / 32 + 6) * 2.0**-24


@pytest.mark.parametrize("d", [64, 128, 192, 256, 384, 448, 512])
@pytest.mark.parametrize("sizes", [[2] * 9, [1, 3, 5, 40], [33, 34], [9]])
def test_scores_of_groups(aps, d, sizes):
    """Groups of near rows: pairs of a group only, each row with 0 to 39 later candidates."""
    import torch

    rng = np.random.default_rng(d + len(sizes))
    q = np.linalg.qr(rng.standard_normal((d, d)))[0][: len(sizes)]
    group = np.repeat(np.arange(len(sizes)), sizes)
    x = q[group] + 0.3 / np.sqrt(d) * rng.standard_normal((group.size, d))
    order = rng.permutation(group.size)
    x, group = (x / np.linalg.norm(x, axis=1, keepdims=True)).astype(np.float32)[order], group[order]
    p, _ = aps.aps_all_pairs_dense(torch.from_numpy(x).cuda(), 0.6)
    try:
        i, j, s = aps.pairs_to_numpy(p)
    finally:
        aps.aps_pairs_free(p)
    full = x.astype(np.float64) @ x.astype(np.float64).T
    wi, wj = np.nonzero(np.triu(group[:, None] == group[None, :], 1))
    assert np.array_equal(i, wi) and np.array_equal(j, wj)
    assert np.all(np.abs(s - full[i, j]) <= (d / 32 + 6) * 2.0**-24)
