"""The resident merge of the workers' row lists (small lists; 33 to 128 workers) against the CPU checker
at the edges of its two forms and of the worker counts, with dropped workers and ids outside the table."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _lists(rng, K, V, sizes):
    parts = [np.sort(rng.choice(V, size=min(n, V), replace=False)).astype(np.int32) for n in sizes]
    return np.concatenate(parts), np.concatenate([[0], np.cumsum([len(p) for p in parts])]).astype(np.int64)


@pytest.mark.parametrize("K,V,total", [
    (1, 5, 1), (2, 40, 33), (3, 1000, 1500), (32, 700, 8000), (5, 1 << 20, 16 * 2048), (5, 1 << 20, 16 * 2048 + 1),
    (33, 90, 2000), (90, 200_000, 60_000), (128, 3000, 120_000), (129, 3000, 20_000), (40, 2_000_000, 900_000),
    (60, 3_000_000, 1_700_000)])  # the last two: 16 and 24 pairs a thread
def test_merge_matches_checker(K, V, total):
    rng = np.random.default_rng(K * 7 + total)
    cuts = np.sort(rng.integers(0, total + 1, size=K - 1))
    uid, wuo = _lists(rng, K, V, np.diff(np.concatenate([[0], cuts, [total]])))
    g = rng.normal(size=(len(uid), 8)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    (ids, agg, n, _, code), names = G.kernels_of(lambda: G.gpu_aggregate(uid, wuo, g, bsz, V))
    assert ("resident_merge" in names) == (K <= 32 and total <= 16 * 2048 or 32 < K <= 128)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids)
    G.close(agg, want)


@pytest.mark.parametrize("K", [6, 70])
def test_dropped_workers_and_foreign_ids(K):
    rng = np.random.default_rng(K)
    V, D = 5000, 8
    uid, wuo = _lists(rng, K, V, [200] * K)
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = [3 + i for i in range(K)]
    dropped = [i % 3 == 1 for i in range(K)]
    agg_ids = torch.zeros(len(uid), dtype=torch.int32, device="cuda")
    agg = torch.zeros(len(uid), D, device="cuda")
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = torch.empty(B.antdt_weighted_aggregate_workspace_bytes(len(uid), D, K), dtype=torch.uint8, device="cuda")
    st = G.new_status()
    B.antdt_weighted_aggregate(bsz, ws, n_rows=V, uniq_ids=G.dev(uid), worker_uniq_offsets=G.dev(wuo),
                               uniq_grads=G.dev(g), agg_ids=agg_ids, agg_grads=agg, n_agg=n, dev_status=st,
                               dropped=dropped)
    assert B.antdt_read_status(st) == 0
    keep = [i for i in range(K) if not dropped[i]]
    kid = np.concatenate([uid[wuo[i]:wuo[i + 1]] for i in keep])
    kg = np.concatenate([g[wuo[i]:wuo[i + 1]] for i in keep])
    want_ids, want = oracle.aggregate_sparse(kid, np.arange(len(keep) + 1, dtype=np.int64) * 200, kg,
                                             np.array([bsz[i] for i in keep], np.int64))
    m = int(n.item())
    assert m == len(want_ids) and np.array_equal(agg_ids[:m].cpu().numpy(), want_ids)
    G.close(agg[:m].cpu().numpy(), want)
    uid[wuo[1] - 1] = V + 3      # the last id of worker 0 lies outside the table: skipped and flagged
    ids, _, _, _, code = G.gpu_aggregate(uid, wuo, g, bsz, V)
    assert code == B.ERR_ID_OUT_OF_RANGE and ids.max() < V


@pytest.mark.parametrize("K,D", [(1, 4), (5, 20), (40, 64), (128, 200)])
def test_sums_by_rows_at_the_capacity(K, D):
    """Short lists are summed row by row: every row kept must be right when the capacity cuts the rest."""
    rng = np.random.default_rng(K)
    uid, wuo = _lists(rng, K, 500, [150] * K)
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = rng.integers(1, 9, size=K)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    for cap in (1, len(want_ids) - 1, len(want_ids)):
        ids, agg, n, _, code = G.gpu_aggregate(uid, wuo, g, bsz, 500, out_cap=cap)
        assert n == len(want_ids) and code == (B.ERR_CAPACITY if cap < n else 0)
        assert np.array_equal(ids, want_ids[:cap])
        G.close(agg, want[:cap])
