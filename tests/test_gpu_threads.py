"""Calls of different shapes from several host threads at once: queries of two indexes with different
tile shapes (whose kernels ask for different amounts of shared memory), batches whose dimension
counts differ. Each call answers as it does alone."""
import threading

import numpy as np
import pytest

import synth

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


def _at_once(jobs, rounds):
    """Each job `rounds` times on a thread of its own, all threads started together."""
    errors, gate = [], threading.Barrier(len(jobs))

    def work(job):
        gate.wait()
        try:
            for _ in range(rounds):
                job()
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors


def test_queries_of_two_tile_shapes_from_two_threads(aps):
    import torch

    rng = np.random.default_rng(101)
    c = synth.sparse_vectors(3000, 500, rng.integers(5, 40, 3000), 1.0, "uniform", 101, rng=rng)
    before, jobs, handles = aps.aps_get_tuning(True), [], []
    try:
        for g in (1, 2, 1, 8):
            aps.aps_set_tuning(aps.aps_get_tuning(), [g] * len(before))
            h = aps.aps_build_index(c.indptr, c.idx, c.val, c.n, c.m, 0.6, aps.QUERYABLE, torch.cuda.Stream())
            handles.append(h)

            def ask(h=h):
                p = aps.aps_query(h, c.indptr[:65], c.idx, c.val, 64, 0.6, aps.HOST_OUTPUT)
                try:
                    return aps.pairs_to_numpy(p)
                finally:
                    aps.aps_pairs_free(p)

            alone = ask()
            assert alone[0].size >= 64

            def same(ask=ask, alone=alone):
                for a, b in zip(ask(), alone):
                    assert np.array_equal(a, b)

            jobs.append(same)
        _at_once(jobs, 300)
    finally:
        aps.aps_set_tuning(aps.aps_get_tuning(), before)
        for h in handles:
            aps.aps_index_free(h)


def test_batches_of_different_dimension_counts_from_two_threads(aps):
    import torch

    rng = np.random.default_rng(102)
    jobs = []
    for m in (200, 57344, 20000, 57000):  # all counted in shared memory: 4 bytes a dimension
        parts = [synth.sparse_vectors(60, m, rng.integers(3, 9, 60), 1.0, "uniform", 102, rng=rng) for _ in range(2)]
        ptr = np.concatenate([parts[0].indptr, parts[0].nnz + parts[1].indptr[1:]])
        csr = [torch.from_numpy(a).cuda() for a in (ptr, *(np.concatenate([getattr(p, k) for p in parts])
                                                           for k in ("idx", "val")))]

        def join(csr=csr, m=m, stream=torch.cuda.Stream()):
            outs, st = aps.aps_batch_all_pairs_csr([0, 60, 120], *csr, [m, m], [0.3, 0.3], 0, stream)
            try:
                return [o.count for o in outs]
            finally:
                for o in outs:
                    aps.aps_pairs_free(o)

        torch.cuda.synchronize()
        alone = join()

        def same(join=join, alone=alone):
            assert join() == alone

        jobs.append(same)
    _at_once(jobs, 1000)
