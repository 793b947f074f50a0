"""The forward that reads bags ahead: bag counts around one wave of lane groups (where it starts), lists that are empty,
shorter and longer than a lane group and than the rows in flight, ids and offsets that are not valid, every row width that
takes it; against the CPU checker.  Inside a step, where bags may go field by field: the same bits."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200.step import DeviceStep, OptConfig, StepBuffers
from tests import gpu_util as G
from tests.test_gpu_parity import _bf16_bits

pytestmark = pytest.mark.gpu
PER_WAVE = 148 * 8 * 256                      # lanes of one resident wave


def _input(rng, n_bags, mean, V, D, bf16):
    lens = rng.poisson(1.25 * mean, size=n_bags)             # a tenth are empty: the mean stays above `mean`
    lens[rng.integers(0, n_bags, size=n_bags // 10)] = 0
    lens[rng.integers(0, n_bags, size=20)] = [1, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 70, 100, 130, 200]
    assert lens.sum() >= mean * n_bags                       # the rule goes by the mean
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, V, size=int(off[-1])).astype(np.int32)
    W = rng.normal(0, 0.01, size=(V, D)).astype(np.float32)
    return _bf16_bits(W) if bf16 else W, ids, off


@pytest.mark.parametrize("D,bf16,lanes,mean", [(128, False, 32, 8), (96, False, 32, 10), (64, False, 16, 6), (48, False, 16, 20),
                                               (32, False, 8, 8), (16, False, 4, 3), (256, True, 32, 16), (128, True, 16, 8),
                                               (64, True, 8, 4), (64, True, 8, 2), (32, True, 4, 3)])
@pytest.mark.parametrize("off_by", [0, 1])
def test_bags(D, bf16, lanes, mean, off_by):
    n_bags = (PER_WAVE // lanes) * (1 + off_by) + off_by
    rng = np.random.default_rng(D + mean + off_by)
    V = 3000
    Wt, ids, off = _input(rng, n_bags, mean, V, D, bf16)
    got, code = G.gpu_fwd(Wt, ids, off)
    assert code == 0 and np.isfinite(got).all()
    pick = np.unique(np.concatenate([[0, n_bags - 1], np.argsort(off[1:] - off[:-1])[-30:], rng.integers(0, n_bags, 3000)]))
    some = np.concatenate([ids[off[b]:off[b + 1]] for b in pick])
    cut = np.concatenate([[0], np.cumsum(off[pick + 1] - off[pick])]).astype(np.int64)
    G.close(got[pick], oracle.embbag_fwd(Wt, some, cut))
    bad = ids.copy()
    bad[off[7]:off[8]] = V                    # skipped and flagged
    bad[-1] = -1
    got2, code = G.gpu_fwd(Wt, bad, off)
    assert code == B.ERR_ID_OUT_OF_RANGE and (off[7] == off[8] or not got2[7].any()) and np.array_equal(got2[8:-40], got[8:-40])
    cut = off.copy()
    cut[n_bags // 2] = -5                     # two bags with bad offsets: empty and flagged
    got3, code = G.gpu_fwd(Wt, ids, cut)
    h = n_bags // 2
    assert code == B.ERR_BAD_OFFSETS and not got3[h - 1:h + 1].any() and np.array_equal(got3[:h - 1], got[:h - 1])


@pytest.mark.parametrize("D,bf16,mean", [(64, False, 9), (64, False, 16), (64, True, 8), (64, True, 16), (32, True, 8), (128, True, 8)])
def test_inside_a_step(D, bf16, mean):
    rng = np.random.default_rng(D + mean)
    F, V, K = 6, 5000, 3
    S = PER_WAVE // (D // (8 if bf16 else 4)) // F + 5
    Wt, ids, off = _input(rng, S * F, mean, V, D, bf16)
    table, ids_t, off_t = G.table_to_dev(Wt), G.dev(ids), G.dev(off)
    buf = StepBuffers(D, K, len(ids), S * F)
    want = torch.zeros(S * F, D, device="cuda")
    B.antdt_embbag_fwd(table, ids_t, off_t, want)
    s0 = torch.ones(V, D, device="cuda")
    step = DeviceStep(buf, table, s0, None, OptConfig(B.OPT_ADAGRAD, 0.01), K, True)
    cuts = [0, S // 2, S // 2 + 3, S]
    step.run(1, ids_t, off_t, F, torch.zeros(S * F, D, device="cuda"), cuts, np.diff(cuts).tolist())
    torch.cuda.synchronize()
    assert int(buf.status) == 0 and torch.equal(buf.pooled[:S * F], want)


def _exact(Wt, ids, bf16):
    """Sums of the rows in 64 bits, and the largest error of a sum of so many terms in 32 bits, in any order."""
    W = ((Wt.astype(np.uint32) << 16).view(np.float32) if bf16 else Wt).astype(np.float64)[ids]
    return W.sum(0), len(ids) * 2.0 ** -24 * np.abs(W).sum(0) + 1e-12


@pytest.mark.parametrize("D,bf16,lanes,mean", [(16, False, 4, 3), (32, False, 8, 8), (64, False, 16, 6), (32, True, 4, 3), (24, True, 4, 4),
                                               (64, True, 8, 4), (128, True, 16, 5), (256, True, 32, 16)])
def test_bags_of_very_many_ids(D, bf16, lanes, mean):
    """Long bags that share a warp with one another and with short and empty ones, in a group's first turn and its last."""
    rng = np.random.default_rng(D + mean)
    wave, V = PER_WAVE // lanes, 3000
    n_bags = wave + 3
    lens = rng.poisson(1.25 * mean, size=n_bags)
    at = np.array([0, 1, 3, 4, 6, 9, wave // 2, wave // 2 + 1, wave // 2 + 5, n_bags - 2, n_bags - 1])
    lens[at] = [256, 5000, 255, 257, 287, 288, 289, 3001, 256, 1024, 20_000]
    lens[[2, 5]] = [0, 1]
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, V, size=int(off[-1])).astype(np.int32)
    W = rng.normal(0, 0.01, size=(V, D)).astype(np.float32)
    Wt = _bf16_bits(W) if bf16 else W
    got, code = G.gpu_fwd(Wt, ids, off)
    assert code == 0
    for b in np.concatenate([np.arange(12), at]):
        want, err = _exact(Wt, ids[off[b]:off[b + 1]], bf16)
        assert (np.abs(got[b] - want) <= err).all(), b
    bad = ids.copy()
    skipped = off[1] + np.array([0, 31, 32, 255, 4999])       # of the bag of 5000: skipped and flagged
    bad[skipped] = [V, -1, V + 7, V, 2**31 - 1]
    got2, code = G.gpu_fwd(Wt, bad, off)
    want, err = _exact(Wt, np.delete(ids[off[1]:off[2]], skipped - off[1]), bf16)
    assert code == B.ERR_ID_OUT_OF_RANGE and (np.abs(got2[1] - want) <= err).all()
    assert np.array_equal(np.delete(got2, 1, 0), np.delete(got, 1, 0))


def test_long_bags_inside_a_step():
    rng = np.random.default_rng(2)
    D, F, V, K = 64, 6, 3000, 3
    S = PER_WAVE // 16 // F + 5
    lens = rng.poisson(20, size=S * F)
    lens[[0, 1, 6, 12, 18, 24, 30, S * F - 7, S * F - 1]] = [256, 3000, 255, 0, 700, 257, 1, 9000, 300]
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, V, size=int(off[-1])).astype(np.int32)
    W = rng.normal(0, 0.01, size=(V, D)).astype(np.float32)
    buf, table, s0 = StepBuffers(D, K, len(ids), S * F), G.dev(W), torch.ones(V, D, device="cuda")
    step = DeviceStep(buf, table, s0, None, OptConfig(B.OPT_ADAGRAD, 0.01), K, True)
    cuts = [0, S // 2, S // 2 + 3, S]
    step.run(1, G.dev(ids), G.dev(off), F, torch.zeros(S * F, D, device="cuda"), cuts, np.diff(cuts).tolist())
    torch.cuda.synchronize()
    got = buf.pooled[:S * F].cpu().numpy()
    assert int(buf.status) == 0
    for b in list(range(40)) + [S * F - 7, S * F - 6, S * F - 1]:
        want, err = _exact(W, ids[off[b]:off[b + 1]], False)
        assert (np.abs(got[b] - want) <= err).all(), b


@pytest.mark.parametrize("D,bf16,lanes,mean,waves", [(16, False, 4, 3, 64), (128, False, 32, 8, 63), (128, False, 32, 8, 64), (128, False, 32, 8, 129)])
def test_many_turns(D, bf16, lanes, mean, waves):
    """Bags on both sides of the counts from which the grid is more than one wave, and not larger any more."""
    n_bags = PER_WAVE // lanes * waves + waves
    rng = np.random.default_rng(waves)
    lens = rng.integers(0, 2 * mean + 2, size=n_bags)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    ids = rng.integers(0, 3000, size=int(off[-1])).astype(np.int32)
    W = rng.normal(0, 0.01, size=(3000, D)).astype(np.float32)
    out, st = torch.full((n_bags, D), float("nan"), device="cuda"), G.new_status()
    B.antdt_embbag_fwd(G.dev(W), G.dev(ids), G.dev(off), out, st)
    assert int(st) == 0 and not out.isnan().any()
    pick = np.unique(np.concatenate([[0, n_bags - 1], rng.integers(0, n_bags, 5000)]))
    some = np.concatenate([ids[off[b]:off[b + 1]] for b in pick])
    cut = np.concatenate([[0], np.cumsum(off[pick + 1] - off[pick])]).astype(np.int64)
    G.close(out[G.dev(pick)].cpu().numpy(), oracle.embbag_fwd(W, some, cut))
