"""The dense part of the aggregation on its side stream (large enough parts, beside a sparse part): sizes
around its tiles, worker counts around its groups of four, workers that count for nothing, a padded stride,
and more workers than the side stream's kernel takes; against the same sum in float64."""
import pytest
import torch

from paper_2404_09679_b200 import binding as B

pytestmark = pytest.mark.gpu
TILE = 768


@pytest.mark.parametrize("K,n,pad,dropped", [
    (1, 1 << 20, 0, ()), (3, TILE * 700, 0, ()), (3, TILE * 700 + 4, 8, (1,)), (4, TILE * 700 - 4, 0, ()),
    (5, TILE * 1000 + 388, 4, (0, 4)), (32, 148 * TILE + 384, 0, (7,)), (33, 148 * TILE + 388, 0, range(4, 9)),
    (128, 20_000, 0, ()), (129, 20_000, 0, ())])
def test_dense_part_beside_a_sparse_part(K, n, pad, dropped):
    assert n * 4 * (K + 1) >= 8 << 20
    gen = torch.Generator("cuda").manual_seed(n)
    dense = torch.randn(K, n + pad, device="cuda", generator=gen)[:, :n]
    out = torch.full((n,), float("nan"), device="cuda")
    uid = torch.arange(K * 3, dtype=torch.int32, device="cuda")
    wuo = torch.arange(K + 1, device="cuda") * 3
    g = torch.ones(K * 3, 4, device="cuda")
    agg_ids, agg = torch.zeros_like(uid), torch.zeros_like(g)
    n_agg, st = torch.zeros(1, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.empty(B.antdt_weighted_aggregate_workspace_bytes(K * 3, 4, K), dtype=torch.uint8, device="cuda")
    bsz = [0 if i % 6 == 5 else 10 + i for i in range(K)]
    drop = [i in dropped for i in range(K)]
    for _ in range(2):
        B.antdt_weighted_aggregate(bsz, ws, n_rows=K * 3, uniq_ids=uid, worker_uniq_offsets=wuo, uniq_grads=g,
                                   agg_ids=agg_ids, agg_grads=agg, n_agg=n_agg, dense_grads=dense, dense_out=out,
                                   dev_status=st, dropped=drop if any(drop) else None)
        copy = out.clone()          # on the caller's stream, right behind the call
    assert B.antdt_read_status(st) == 0
    w = torch.tensor([0.0 if d else float(b) for b, d in zip(bsz, drop)], dtype=torch.float64, device="cuda")
    want = ((w / w.sum())[:, None] * dense.double()).sum(0)
    assert torch.allclose(copy.double(), want, rtol=1e-5, atol=1e-6)
