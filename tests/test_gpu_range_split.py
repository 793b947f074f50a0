"""The range merge's boundaries: lists on both sides of the count from which one lane looks for a boundary instead of
eight, list lengths around powers of nine (probes of eight lanes), empty lists, dense and sparse ones, a table whose last
range is a part of one, ids at the ends of the table; sums by rows on both sides of their rule; and ranges of as many entries as the emit kernel's CTA keeps in registers or puts
in order in shared memory.  Against the CPU checker."""
import numpy as np
import pytest

import oracle
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _check(rng, V, sizes, D, ends=True):
    parts = []
    for n in sizes:
        p = np.sort(rng.choice(V, size=min(n, V), replace=False)).astype(np.int32) if n else np.zeros(0, np.int32)
        if ends and len(p) > 2:
            p[0], p[-1] = 0, V - 1
            p = np.unique(p)
        parts.append(p)
    uid = np.concatenate(parts)
    wuo = np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = rng.integers(1, 50, size=len(sizes))
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    ids, agg, n, _, code = G.gpu_aggregate(uid, wuo, g, bsz, V)
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)


@pytest.mark.parametrize("V", [700_000, 4096 * 190, 4096 * 3200, 4096 * 4000 + 1])
def test_boundaries(V):
    rng = np.random.default_rng(V % 1000)
    # 16 workers: 4096 * 3200 rows have 51 k boundaries, more than eight lanes look for together
    _check(rng, V, [0, 1, 2, 8, 9, 10, 80, 81, 82, 729, 6561, 6560, 59_049, 0, 70_001, 0], 4)


@pytest.mark.parametrize("K,n,D,V", [(32, 1200, 4, 9000), (2, 65_536, 64, 65_536), (2, 65_537, 64, 70_000), (3, 30_000, 20, 45_000),
                                     (3, 30_001, 20, 45_000), (1, 40_000, 200, 2_000_000), (32, 2600, 100, 300_000)])
def test_sums_by_rows_and_by_tiles(K, n, D, V):
    rng = np.random.default_rng(K * n)
    _check(rng, V, [n] * K, D, ends=False)


# many workers that list the same rows: each row's sum would be one lane group's chain
@pytest.mark.parametrize("K,by_rows", [(16, True), (17, False), (32, False)])
def test_many_workers_rows_are_summed_by_tiles(K, by_rows):
    rng = np.random.default_rng(K)
    uid = np.concatenate([np.sort(rng.choice(6000, size=3000, replace=False)) for _ in range(K)]).astype(np.int32)
    wuo = np.arange(K + 1, dtype=np.int64) * 3000
    g = rng.normal(size=(len(uid), 20)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    (ids, agg, n, _, code), names = G.kernels_of(lambda: G.gpu_aggregate(uid, wuo, g, bsz, 1_000_000))
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)
    assert "agg_range_emit" in names and ("agg_fixup" not in names) == by_rows


# entries of the first range around 4 and 8 per thread; more than the staged slots (1536 here) in the last three
@pytest.mark.parametrize("D", [4, 132])
@pytest.mark.parametrize("K", [16, 17, 32])
@pytest.mark.parametrize("n", [1023, 1024, 1025, 2048, 2049, 4097, 30_000])
def test_entries_per_range(n, K, D):
    rng = np.random.default_rng(n + K)
    V = 4096 * 60 + 7
    parts = []
    for w in range(K):
        k = min(4096, n // K + (w < n % K))
        parts.append(np.sort(np.concatenate([rng.choice(4096, size=k, replace=False),
                                             4096 + rng.choice(V - 4096, size=66_000 // K, replace=False)])).astype(np.int32))
    uid = np.concatenate(parts)
    wuo = np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    ids, agg, m, _, code = G.gpu_aggregate(uid, wuo, g, bsz, V)
    assert code == 0 and m == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)
