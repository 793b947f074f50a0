"""Ids outside the table at the end of the workers' lists (more entries than the resident merge takes): they are
flagged and skipped, and the rows inside the table get their own sums whatever the workspace held before."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("update", [False, True])
@pytest.mark.parametrize("K,V,per,foreign", [(2, 20_000, 18_000, [20_000, -1]), (5, 50_003, 9000, [50_003, 50_004, 61_440]),
                                             (32, 4000, 1500, [4000, 4095, 4096, 2**31 - 1])])
def test_rows_of_the_table_get_their_own_sums(K, V, per, foreign, update):
    rng = np.random.default_rng(K)
    D = 8
    clean = [np.sort(rng.choice(V, size=per, replace=False)).astype(np.int32) for _ in range(K)]
    for c in clean[1:]:
        c[-1] = V - 1                                  # the last row of the table has the last slots
    lists = [np.concatenate([c, np.array(foreign[:1 + i % len(foreign)], np.int64).astype(np.int32)])
             for i, c in enumerate(clean)]
    uid = np.concatenate(lists)
    wuo = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(np.int64)
    assert len(uid) > 16 * 2048
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    inside = (uid >= 0) & (uid < V)
    bsz = rng.integers(1, 50, size=K)
    cw = np.concatenate([[0], np.cumsum([len(c) for c in clean])]).astype(np.int64)
    want_ids, want = oracle.aggregate_sparse(uid[inside], cw, g[inside], bsz.astype(np.int64))
    uid_t, wuo_t, g_t, st = G.dev(uid), G.dev(wuo), G.dev(g), G.new_status()
    g_t[G.dev(~inside)] = float("nan")                 # nothing of a skipped element may reach a row
    n = torch.zeros(1, dtype=torch.int64, device="cuda")
    agg_ids = torch.zeros(len(uid), dtype=torch.int32, device="cuda")
    agg = torch.zeros(len(uid), D, device="cuda")
    table, s0 = torch.zeros(V, D, device="cuda"), torch.zeros(V, D, device="cuda")
    size = B.antdt_weighted_aggregate_workspace_bytes(len(uid), D, K)
    for fill in (0, 0xFF, 0x55):
        ws = torch.full((size,), fill, dtype=torch.uint8, device="cuda")
        ws.view(torch.int32)[:] = len(uid) - 1 if fill == 0x55 else ws.view(torch.int32)  # a position of a skipped element
        s0.zero_()
        args = dict(uniq_ids=uid_t, worker_uniq_offsets=wuo_t, uniq_grads=g_t, agg_ids=agg_ids, n_agg=n, dev_status=st)
        if update:                                     # Adagrad at rate 0: s0 is the square of the row's sum
            B.antdt_aggregate_update(bsz.tolist(), ws, table, B.OPT_ADAGRAD, 0.0, 1e-8, 0.0, 0.0, 1, s0, **args)
        else:
            B.antdt_weighted_aggregate(bsz.tolist(), ws, n_rows=V, agg_grads=agg, **args)
        assert B.antdt_read_status(st) == B.ERR_ID_OUT_OF_RANGE
        m = int(n.item())
        assert m == len(want_ids) and np.array_equal(agg_ids[:m].cpu().numpy(), want_ids)
        if update:
            G.close(s0[agg_ids[:m].long()].cpu().numpy(), want.astype(np.float64) ** 2, rtol=3e-5)
        else:
            G.close(agg[:m].cpu().numpy(), want)
