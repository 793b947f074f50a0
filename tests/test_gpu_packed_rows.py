"""Rows whose vectors do not fill a power of two of lanes: forward, sums and updates with the rows packed lane by
lane, around CTA edges (a row that begins in one warp and ends in the next, threads left over at a CTA's end, a
last CTA with one row); against the CPU checker, and on every path the rows behind the last one stay untouched."""
import numpy as np
import pytest

import oracle
from tests import gpu_util as G
from tests import test_gpu_fused_update as fused
from tests.test_gpu_parity import _bf16_bits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,bf16,hi", [(20, False, 6), (36, False, 3), (40, False, 9), (68, False, 2), (80, False, 5),
                                       (40, True, 6), (72, True, 3), (136, True, 2), (160, True, 4)])
@pytest.mark.parametrize("n_bags", [1, 51, 52, 1000, 148 * 8 * 51 * 8 + 1])
def test_forward(D, bf16, hi, n_bags):
    if n_bags > 100_000 and D > 40:
        n_bags = 148 * 8 * (256 * (8 if bf16 else 4) // D) * 8 + 1      # the first count that is strided over
    rng = np.random.default_rng(D + n_bags)
    V = 2000
    W = rng.normal(0, 0.01, size=(V, D)).astype(np.float32)
    Wt = _bf16_bits(W) if bf16 else W
    off = np.concatenate([[0], np.cumsum(rng.integers(0, hi + 1, size=n_bags))]).astype(np.int64)
    ids = rng.integers(0, V, size=off[-1]).astype(np.int32)
    got, code = G.gpu_fwd(Wt, ids, off)
    assert code == 0 and np.isfinite(got).all()
    pick = np.unique(np.concatenate([[0, n_bags - 1], rng.integers(0, n_bags, 3000)]))
    some = np.concatenate([ids[off[b]:off[b + 1]] for b in pick])
    cut = np.concatenate([[0], np.cumsum(off[pick + 1] - off[pick])]).astype(np.int64)
    G.close(got[pick], oracle.embbag_fwd(Wt, some, cut))


@pytest.mark.parametrize("opt", ["adagrad", "adam"])
@pytest.mark.parametrize("D,bf16", [(12, False), (20, False), (24, True), (40, False), (48, False), (96, True),
                                    (112, False)])
@pytest.mark.parametrize("n", [1, 11, 2001])
def test_sparse_update(opt, D, bf16, n):
    rng = np.random.default_rng(D + n)
    V = 5000
    W = rng.normal(0, 0.5, size=(V, D)).astype(np.float32)
    W = _bf16_bits(W) if bf16 else W
    ids = np.sort(rng.choice(V, size=n, replace=False)).astype(np.int32)
    g = rng.normal(size=(n, D)).astype(np.float32)
    s0 = np.abs(rng.normal(size=(V, D))).astype(np.float32)
    s1 = np.abs(rng.normal(size=(V, D))).astype(np.float32) if opt == "adam" else None
    ref = [W.copy(), s0.copy(), None if s1 is None else s1.copy()]
    oracle.sparse_opt_update(ref[0], ids, g, opt, 0.05, 1e-8, 0.9, 0.999, 3, ref[1], ref[2])
    t, d0, d1, code = G.gpu_update(W, ids, g, opt, 0.05, 1e-8, 0.9, 0.999, 3, s0, s1)
    assert code == 0
    G.close(d0, ref[1])
    if s1 is not None:
        G.close(d1, ref[2])
    if bf16:
        G.close(_f32(t), _f32(ref[0]), rtol=G.BF16_RTOL)
    else:
        G.close(t, ref[0])
    rest = np.setdiff1d(np.arange(V), ids)
    assert np.array_equal(t[rest], W[rest]) and np.array_equal(d0[rest], s0[rest])


def _f32(bits):
    return (bits.astype(np.uint32) << 16).view(np.float32)


@pytest.mark.parametrize("D,K,n_per", [(20, 5, 40), (40, 3, 700), (96, 8, 333), (12, 2, 5)])
def test_sums_of_short_lists(D, K, n_per):
    rng = np.random.default_rng(D + K)
    V = 3000
    uid, wuo = fused._lists(rng, K, V, n_per, rng.integers(0, V, size=50))
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz)
    ids, agg, n, _, code = G.gpu_aggregate(uid, wuo, g, bsz, V)
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)


@pytest.mark.parametrize("opt,D,bf16,K", [("adagrad", 20, False, 5), ("adagrad", 48, False, 3), ("adagrad", 24, True, 8),
                                          ("adam", 40, False, 7), ("adam", 40, True, 32), ("adagrad", 96, False, 16)])
def test_one_pass_server_step(opt, D, bf16, K):
    fused.test_fused_aggregate_update_matches_the_checkers_two_steps(opt, D, bf16, K, K == 3)
