"""The walk's fix-up inside its last CTA (2 to 24 stretches of 16-entry tiles): runs that leave their
stretch from the tile of its last lane group, time after time on a cleared workspace.  A row whose task is
missed stays NaN, a task taken before its words are stored writes row 0 of the wrong stretch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,stretches,K", [(4, 2, 1), (8, 24, 3), (16, 2, 1), (16, 23, 5), (64, 24, 1), (96, 13, 2),
                                           (128, 2, 1), (128, 24, 4), (512, 24, 1)])
def test_every_run_that_leaves_a_stretch_is_written(D, stretches, K):
    lanes = 1
    while lanes < min(32, D // 4):
        lanes *= 2
    span = 16 * (256 // lanes)                      # entries of a stretch
    n = stretches * span - 5
    rng = np.random.default_rng(D + stretches)
    # a run starts in the last tile of every stretch (and a few elsewhere), so each stretch leaves a task
    starts = np.concatenate([np.arange(1, stretches) * span - rng.integers(1, 16, size=stretches - 1),
                             rng.integers(1, n, size=stretches)])
    ids = np.zeros(n, np.int64)
    ids[starts] = 1
    ids = np.cumsum(ids).astype(np.int32)
    V, off = int(ids[-1]) + 1, np.arange(n + 1, dtype=np.int64)
    wso = np.concatenate([[0], np.sort(rng.integers(0, n + 1, size=K - 1)), [n]])
    dY = rng.normal(size=(n, D)).astype(np.float32)
    want = oracle.embbag_bwd_dedup(ids, off, 1, dY, V, wso)
    nu = len(want["uniq_ids"])
    ids_t, off_t, dY_t, st = G.dev(ids), G.dev(off), G.dev(dY), G.new_status()
    uid = torch.zeros(n, dtype=torch.int32, device="cuda")
    wuo, so = torch.zeros(K + 1, dtype=torch.int64, device="cuda"), torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    occ = torch.zeros(n, dtype=torch.int32, device="cuda")
    ug = torch.empty(n, D, device="cuda")
    ws = torch.empty(B.antdt_embbag_bwd_dedup_workspace_bytes(n, n, D, K), dtype=torch.uint8, device="cuda")
    first = None
    for _ in range(60):
        ws.zero_()
        ug.fill_(float("nan"))
        B.antdt_embbag_bwd_dedup(ids_t, off_t, 1, dY_t, V, wso.tolist(), uid, wuo, so, occ, ug, ws, st)
        if first is None:
            first = ug[:nu].clone()
        assert torch.equal(ug[:nu], first)
    assert B.antdt_read_status(st) == 0
    # sums of at most n fp32 terms of size 1 in another order: n * 2^-24 of their absolute sum, / b_w
    G.close(first.cpu().numpy(), want["uniq_grads"], atol=3e-6)
