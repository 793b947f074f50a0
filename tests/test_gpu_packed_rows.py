"""Rows whose vectors do not fill a power of two of lanes: forward, sums and updates with the rows packed lane by
lane, around CTA edges (a row that begins in one warp and ends in the next, threads left over at a CTA's end, a
last CTA with one row); against the CPU checker, and on every path the rows behind the last one stay untouched."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200.step import DeviceStep, OptConfig, StepBuffers
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
    _check_forward(D, bf16, hi, n_bags)


# Rows are packed from so many bags on: tenths of one resident wave of unpacked lane groups.
def _line(D, bf16):
    lanes = 1 << (D // (8 if bf16 else 4) - 1).bit_length()
    return -(-148 * 8 * (256 // lanes) * (25 if bf16 else 12) // 10)


@pytest.mark.parametrize("D,bf16,hi", [(20, False, 6), (40, False, 20), (80, False, 5), (40, True, 6), (72, True, 20), (160, True, 4)])
@pytest.mark.parametrize("over", ["below", "at", "one row in the last CTA", "a full last CTA"])
def test_forward_around_the_count_from_which_rows_are_packed(D, bf16, hi, over):
    line, per = _line(D, bf16), 256 // (D // (8 if bf16 else 4))
    full = -(-line // per) * per
    _check_forward(D, bf16, hi, {"below": line - 1, "at": line, "one row in the last CTA": full + 1, "a full last CTA": full}[over])


@pytest.mark.parametrize("D,bf16", [(20, False), (36, False), (80, False), (40, True), (160, True)])
@pytest.mark.parametrize("F", [3, 7])
def test_forward_inside_a_step(D, bf16, F):
    """Nine ids a bag: one field at a time, CTAs of consecutive samples, the last of them with a part of its rows."""
    rng = np.random.default_rng(D + F)
    V, K, S = 3000, 3, _line(D, bf16) // F + 2
    off = np.concatenate([[0], np.cumsum(rng.integers(0, 19, size=S * F) + (np.arange(S * F) % 64 == 5))]).astype(np.int64)
    assert 8 * S * F <= off[-1]                        # the rule of field order
    ids = rng.integers(0, V, size=off[-1]).astype(np.int32)
    W = rng.normal(0, 0.01, size=(V, D)).astype(np.float32)
    Wt = _bf16_bits(W) if bf16 else W
    buf, table, s0 = StepBuffers(D, K, len(ids), S * F), G.table_to_dev(Wt), torch.ones(V, D, device="cuda")
    ids_t, off_t, dY = G.dev(ids), G.dev(off), torch.zeros(S * F, D, device="cuda")
    buf.pooled.fill_(float("nan"))
    step = DeviceStep(buf, table, s0, None, OptConfig(B.OPT_ADAGRAD, 0.01), K, True)
    cuts = [0, S // 2, S // 2 + 3, S]
    step.run(1, ids_t, off_t, F, dY, cuts, np.diff(cuts).tolist())
    torch.cuda.synchronize()
    assert int(buf.status) == 0
    G.close(buf.pooled[:S * F].cpu().numpy(), oracle.embbag_fwd(Wt, ids, off))


def _check_forward(D, bf16, hi, n_bags):
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
