"""The merge of 33 to 128 workers' lists: empty lists and lists of one id, wide gaps and dense stretches, lists that pile up
on a few hot rows, dropped workers, ids outside the table, a capacity that cuts rows off, lists in no order.  Against the CPU
checker.  The sorts' time does not depend on how the ids lie; a merge by ranges of row ids, one CTA each, takes up to four times
theirs where the lists pile up, so none of these may take it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _lists(rng, K, V, per):
    """Lists of all sorts: spread, empty, of one id, a dense stretch with a far id on either side, the table's ends."""
    parts = []
    for w in range(K):
        kind = w % 6
        if kind == 1:
            p = np.zeros(0, np.int64)
        elif kind == 2:
            p = rng.integers(0, V, size=1)
        elif kind == 3:
            at = int(rng.integers(0, max(1, V - per)))
            p = np.concatenate([np.arange(at, min(V, at + per)), [0, V - 1]])
        else:
            p = rng.choice(V, size=min(V, per + w), replace=False)
        parts.append(np.unique(p).astype(np.int32))
    return parts


def _join(parts):
    return np.concatenate(parts), np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)


def _aggregate(uid, wuo, g, bsz, V, dropped=None, out_cap=None, fill=0xAB):
    D, K, cap = g.shape[1], len(bsz), len(uid) if out_cap is None else out_cap
    ids = torch.full((max(cap, 1),), -1, dtype=torch.int32, device="cuda")
    agg = torch.full((max(cap, 1), D), float("nan"), device="cuda")
    n, st = torch.zeros(1, dtype=torch.int64, device="cuda"), G.new_status()
    ws = torch.full((B.antdt_weighted_aggregate_workspace_bytes(len(uid), D, K),), fill, dtype=torch.uint8, device="cuda")
    _, names = G.kernels_of(lambda: B.antdt_weighted_aggregate(
        [int(b) for b in bsz], ws, n_rows=V, uniq_ids=G.dev(uid), worker_uniq_offsets=G.dev(wuo), uniq_grads=G.dev(g),
        agg_ids=ids[:cap], agg_grads=agg[:cap], n_agg=n, dev_status=st, dropped=dropped))
    code, m = B.antdt_read_status(st), int(n.item())
    assert "agg_range_emit" not in names and ("resident_merge" in names) == (len(uid) <= 1_800_000)
    k = min(m, cap)
    return ids[:k].cpu().numpy(), agg[:k].cpu().numpy(), m, code


@pytest.mark.parametrize("K,V,per,D", [(33, 20_000, 3000, 8), (64, 100_001, 4000, 4), (65, 1024 * 300, 3000, 20), (96, 2048 * 500 + 1, 2000, 8),
                                       (97, 1_000_000, 3000, 16), (128, 2047, 1500, 8), (128, 1_200_000, 2500, 4), (128, 3_000_000, 6000, 4), (90, 30_000, 2500, 8),
                                       (40, 1_000_000, 2000, 8), (64, 4_000_000, 45_000, 4)])
def test_matches_checker(K, V, per, D):
    rng = np.random.default_rng(K + V)
    parts = _lists(rng, K, V, per)
    uid, wuo = _join(parts)
    assert len(uid) > 16 * 2048
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    ids, agg, n, code = _aggregate(uid, wuo, g, bsz, V)
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)
    cap = len(want_ids) // 2
    ids, agg, n, code = _aggregate(uid, wuo, g, bsz, V, out_cap=cap)
    assert code == B.ERR_CAPACITY and n == len(want_ids) and np.array_equal(ids, want_ids[:cap])
    G.close(agg, want[:cap])
    # every third worker dropped: as if its list were not there
    dropped = [i % 3 == 1 for i in range(K)]
    keep = [i for i in range(K) if not dropped[i]]
    kid, kwuo = _join([parts[i] for i in keep])
    kg = np.concatenate([g[wuo[i]:wuo[i + 1]] for i in keep])
    want_ids, want = oracle.aggregate_sparse(kid, kwuo, kg, bsz[keep].astype(np.int64))
    ids, agg, n, code = _aggregate(uid, wuo, g, bsz, V, dropped=dropped)
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)


# a table per field, ids by frequency: all lists begin with the fields' hot rows
@pytest.mark.parametrize("K,V,F,n", [(100, 1_000_000, 1, 4500), (60, 200_000, 4, 4000), (90, 390_000, 39, 12_000)])
def test_lists_that_pile_up(K, V, F, n):
    rng = np.random.default_rng(K)
    per = V // F
    parts = []
    for _ in range(K):
        rank = np.minimum((per ** rng.random(n)).astype(np.int64), per) - 1
        parts.append(np.unique(rng.integers(0, F, size=n) * per + rank).astype(np.int32))
    uid, wuo = _join(parts)
    g = rng.normal(size=(len(uid), 8)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    ids, agg, m, code = _aggregate(uid, wuo, g, bsz, V)
    assert code == 0 and m == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)


@pytest.mark.parametrize("K,V", [(40, 50_003), (100, 20_000)])
def test_ids_outside_the_table_and_lists_in_no_order(K, V):
    rng = np.random.default_rng(K)
    parts = _lists(rng, K, V, 1800)
    foreign = [V, V + 1, 61_440, 2**31 - 1, -1]
    lists = [np.concatenate([p, np.array(foreign[:w % 6], np.int64).astype(np.int32)]) for w, p in enumerate(parts)]
    uid, wuo = _join(lists)
    g = rng.normal(size=(len(uid), 8)).astype(np.float32)
    inside = (uid >= 0) & (uid < V)
    bsz = rng.integers(1, 50, size=K)
    cuid, cwuo = _join(parts)
    want_ids, want = oracle.aggregate_sparse(cuid, cwuo, g[inside], bsz.astype(np.int64))
    cg = g[inside]
    g[~inside] = np.nan                                # nothing of a skipped element may reach a row
    for fill in (0, 0xFF):
        ids, agg, n, code = _aggregate(uid, wuo, g, bsz, V, fill=fill)
        assert code == B.ERR_ID_OUT_OF_RANGE and n == len(want_ids) and np.array_equal(ids, want_ids)
        G.close(agg, want)
    for w in range(K):                                 # every list in an order of its own: the same sums
        order = cwuo[w] + rng.permutation(cwuo[w + 1] - cwuo[w])
        cuid[cwuo[w]:cwuo[w + 1]], cg[cwuo[w]:cwuo[w + 1]] = cuid[order], cg[order]
    ids, agg, n, code = _aggregate(cuid, cwuo, cg, bsz, V)
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)
    cuid[cwuo[4]:cwuo[5]] = cuid[cwuo[4]]              # one id over and over
    assert _aggregate(cuid, cwuo, cg, bsz, V)[3] == B.ERR_BAD_OFFSETS
