"""Bag of every occurrence before the multi-kernel sort (129 workers: more than the resident sort takes): empty bags in rows,
bags that begin or end at a turn of 128 slots or a window of 1024, bags over several windows, short ones, ragged ends.  Against
the CPU checker.  And bad offsets in one group of 32 bags of a warp's four: the bags of the other three get their occurrences."""
import numpy as np
import pytest

from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _check_bwd

pytestmark = pytest.mark.gpu

EDGES = [0, 0, 1, 2, 3, 4, 5, 127, 128, 129, 1022, 1023, 1024, 1025, 2047, 2049, 5000]


@pytest.mark.parametrize("make", ["edges", "short", "sparse", "ones", "long"])
@pytest.mark.parametrize("shift", [0, 1, 3])
def test_bags_of_all_lengths(make, shift):
    rng = np.random.default_rng(shift)
    K, per = 129, 5 + shift
    n = K * per
    lens = {"edges": lambda: rng.choice(EDGES, size=n), "short": lambda: rng.integers(0, 9, size=n),
            "sparse": lambda: (rng.random(n) < 0.02) * rng.integers(1, 300, size=n), "ones": lambda: np.ones(n, np.int64),
            "long": lambda: np.where(np.arange(n) % 128 == 77, 20_011, 0)}[make]()
    lens[0] = shift                                    # what follows begins off the 16-byte grid
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, 50_000, size=int(off[-1])).astype(np.int32)
    dY = rng.normal(size=(n, 4)).astype(np.float32)
    _check_bwd(ids, off, 1, dY, 50_000, np.arange(K + 1, dtype=np.int64) * per)


@pytest.mark.parametrize("group", [0, 1, 2, 3, 5])
@pytest.mark.parametrize("off_by", [0, 17, 31])
def test_good_groups_beside_a_bad_one(group, off_by):
    rng = np.random.default_rng(group * 32 + off_by)
    K, per = 129, 32                                   # a worker to a group, four of them to a warp
    n = K * per
    lens = rng.choice([0, 1, 2, 5, 40], size=n)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, 500, size=int(off[-1])).astype(np.int32)
    dY = rng.normal(size=(n, 4)).astype(np.float32)
    wso = np.arange(K + 1, dtype=np.int64) * per
    want = G.gpu_bwd(ids, off, 1, dY, 500, wso)
    assert want["status"] == 0
    at = group * 32 + off_by
    cut = off.copy()
    cut[at + (1 if off_by == 0 else 0)] = -3           # (not a group's first offset, which is the last one of the group before)
    got = G.gpu_bwd(ids, cut, 1, dY, 500, wso)
    assert got["status"] == B.ERR_BAD_OFFSETS and np.array_equal(got["uniq_ids"], want["uniq_ids"])
    wuo = want["worker_uniq_offsets"]
    assert np.array_equal(got["worker_uniq_offsets"], wuo)
    same = np.ones(len(want["uniq_ids"]), bool)
    same[wuo[group]:wuo[group + 1]] = False            # the bad group's occurrences are in no bag
    assert np.array_equal(got["uniq_grads"][same], want["uniq_grads"][same])
