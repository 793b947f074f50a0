"""The forward whose lane groups stride over the bags: bag counts on both sides of the wave counts where it
starts and where it takes a second wave, for bags just below and at the length where each row width stops
striding; against the CPU checker."""
import numpy as np
import pytest

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _bf16_bits

pytestmark = pytest.mark.gpu
PER_WAVE = 148 * 8 * 256                      # lanes of one resident wave


@pytest.mark.parametrize("D,bf16,lanes,waves,off_by,lo,hi", [
    (128, False, 32, 8, -1, 6, 14), (128, False, 32, 8, 0, 6, 14), (96, False, 32, 15, 1, 0, 20),
    (64, False, 16, 8, 0, 4, 16), (128, True, 16, 8, 3, 0, 9), (32, False, 8, 8, 1, 5, 10),
    (32, False, 8, 8, 1, 6, 10), (8, True, 1, 8, 0, 1, 1),
    (128, False, 32, 8, 0, 14, 16), (128, False, 32, 8, 0, 16, 16), (64, False, 16, 8, 2, 13, 18),
    (32, False, 8, 8, 1, 3, 8), (16, False, 4, 8, 0, 1, 4), (16, False, 4, 8, 0, 3, 3), (8, False, 2, 8, 0, 1, 2),
    (256, True, 32, 8, 1, 2, 12), (128, True, 16, 8, 0, 4, 6), (64, True, 8, 15, 1, 1, 6), (64, True, 8, 8, 0, 4, 4),
    (32, True, 4, 8, 0, 1, 3)])
def test_strided_bags(D, bf16, lanes, waves, off_by, lo, hi):
    n_bags = waves * (PER_WAVE // lanes) + off_by
    rng = np.random.default_rng(D + hi + off_by)
    V = 3000
    W = rng.normal(0, 0.01, size=(V, D)).astype(np.float32)
    Wt = _bf16_bits(W) if bf16 else W
    off = np.concatenate([[0], np.cumsum(rng.integers(lo, hi + 1, size=n_bags))]).astype(np.int64)
    ids = rng.integers(0, V, size=off[-1]).astype(np.int32)
    got, code = G.gpu_fwd(Wt, ids, off)
    assert code == 0
    pick = np.unique(np.concatenate([[0, n_bags - 1], rng.integers(0, n_bags, 4000)]))
    some = np.concatenate([ids[off[b]:off[b + 1]] for b in pick])
    cut = np.concatenate([[0], np.cumsum(off[pick + 1] - off[pick])]).astype(np.int64)
    G.close(got[pick], oracle.embbag_fwd(Wt, some, cut))
    assert np.isfinite(got).all()             # every bag was written (the output starts as NaN)
    ids[-1] = V                               # the last group's last turn flags a bad id
    if off[-1] > off[-2]:
        assert G.gpu_fwd(Wt, ids, off)[1] == B.ERR_ID_OUT_OF_RANGE
