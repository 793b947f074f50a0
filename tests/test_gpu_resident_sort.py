"""The resident sort of the backward (one kernel: a cluster of CTAs, or one CTA per SM) against the CPU
checker at the sizes where its layout changes: empty and one-occurrence workers, the edges of a warp,
a CTA and the cluster form, the largest input it takes and one more, 1 to 129 workers."""
import numpy as np
import pytest

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _check(lens, wso, F, V, D, rng, hot=0.3):
    """lens: bag lengths, sample-major; a share `hot` of the ids is one row."""
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, V, size=int(off[-1])).astype(np.int32)
    ids[rng.random(ids.size) < hot] = V // 3
    dY = rng.normal(size=(len(lens), D)).astype(np.float32)
    wso = np.asarray(wso, np.int64)
    got = G.gpu_bwd(ids, off, F, dY, V, wso)
    want = oracle.embbag_bwd_dedup(ids, off, F, dY, V, wso)
    assert got["status"] == 0
    for k in ("worker_uniq_offsets", "uniq_ids", "seg_offsets", "sorted_occ"):
        assert np.array_equal(got[k], want[k]), k
    G.close(got["uniq_grads"], want["uniq_grads"], atol=3e-6)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 511, 513, 1023, 1025, 4095, 4097, 8193, 16_385, 32_768, 32_769, 110_000, 400_001])
def test_one_worker_of_every_size_class(n):
    rng = np.random.default_rng(n)
    lens = np.ones(n, np.int64)
    lens[rng.integers(0, n, size=n // 4)] = 0              # empty bags at the ends and in runs
    if n > 64:
        lens[10:42] = 0
        lens[n // 2] = n // 8                              # a bag that spans CTAs
    if lens.sum() == 0:
        lens[0] = 1
    _check(lens, [0, n], 1, 5_000_000, 8, rng)


@pytest.mark.parametrize("K,S,V", [(3, 7, 2), (32, 640, 1 << 20), (33, 700, 900), (90, 9000, 100_000), (128, 40_000, 5000),
                                   (129, 3000, 50), (200, 1000, 3)])
def test_many_workers_with_empty_and_uneven_parts(K, S, V):
    rng = np.random.default_rng(K)
    cuts = np.sort(rng.integers(0, S + 1, size=K - 1))
    lens = rng.integers(0, 6, size=S * 3)
    _check(lens, np.concatenate([[0], cuts, [S]]), 3, V, 4, rng)


@pytest.mark.parametrize("V", [1, 200, 511, 512, 70_000, 3_000_000, (1 << 31) - 1])
def test_unequal_workers_and_table_sizes(V):
    # equal sample counts, but worker 1 holds nearly every occurrence; 1 to 4 passes
    rng = np.random.default_rng(V % 1000)
    lens = np.concatenate([rng.integers(0, 3, size=4000), rng.integers(20, 60, size=4000), np.zeros(4000, np.int64)])
    _check(lens, [0, 2000, 4000, 6000], 2, V, 8, rng)


@pytest.mark.parametrize("extra", [0, 1])
def test_the_largest_input_and_the_one_after_it(extra):
    rng = np.random.default_rng(9)
    n = 148 * 512 * 24 + extra                 # one more goes to the multi-kernel sort
    lens = np.full(n // 8, 8, np.int64)
    lens[0] += n - lens.sum()
    B.antdt_profile_enable(True)
    _check(lens, [0, len(lens) // 3, len(lens)], 1, 40_000, 4, rng, hot=0.05)
    ran = set(B.antdt_profile_get())
    B.antdt_profile_enable(False)
    assert ("resident_sort" in ran) == (extra == 0) and ("radix_scatter" in ran) == (extra == 1)


@pytest.mark.parametrize("K,n", [(1, 148 * 512 * 24), (8, 148 * 512 * 17 + 31), (9, 148 * 512 * 9 - 33), (2, 148 * 512 * 4 + 1)])
def test_shares_of_the_warps_and_ways_to_rank_by_worker(K, n):
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 5, size=n // 2)
    lens[-1] += max(0, n - lens.sum())
    lens[np.cumsum(lens) > n] = 0
    lens[0] += n - lens.sum()
    cuts = np.sort(rng.integers(0, len(lens) + 1, size=K - 1))
    _check(lens, np.concatenate([[0], cuts, [len(lens)]]), 1, 300_000, 4, rng, hot=0.1)
