"""Calls on a stream that has only some of the device's SMs (a green context's): the resident sort and merge,
whose CTAs must all be on the GPU at once, are refused there and the kernels that do not need it take over,
with the same results.  (Sizes beyond one cluster.)"""
import numpy as np
import pytest
import torch

import oracle
from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_two_trainers import same, trainers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    d = pytest.importorskip("cuda.bindings.driver")

    def ok(r):
        assert r[0] == d.CUresult.CUDA_SUCCESS, r
        return r[1] if len(r) == 2 else r[1:]

    torch.zeros(1, device="cuda")
    dev = ok(d.cuDeviceGet(0))
    sms = ok(d.cuDeviceGetDevResource(dev, d.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    groups, _, _ = ok(d.cuDevSmResourceSplitByCount(1, sms, 0, 64))
    desc = ok(d.cuDevResourceGenerateDesc([groups[0]], 1))
    ctx = ok(d.cuGreenCtxCreate(desc, dev, d.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    raw = ok(d.cuGreenCtxStreamCreate(ctx, d.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    yield torch.cuda.ExternalStream(int(raw))
    torch.cuda.synchronize()
    B.antdt_bsp_step_graph_reset()
    d.cuStreamDestroy(raw)
    d.cuGreenCtxDestroy(ctx)


def _ran(fn, stream):
    with torch.cuda.stream(stream):
        return G.kernels_of(fn)


@pytest.mark.parametrize("n,K,resident", [(60_000, 3, True), (400_000, 3, False), (1_700_000, 2, False)])
def test_backward(stream, n, K, resident):
    rng = np.random.default_rng(n)
    off, V = np.arange(n + 1, dtype=np.int64), 50_000
    ids = rng.integers(0, V, size=n).astype(np.int32)
    dY = rng.normal(size=(n, 8)).astype(np.float32)
    wso = np.array([n * i // K for i in range(K + 1)], np.int64)
    got, names = _ran(lambda: G.gpu_bwd(ids, off, 1, dY, V, wso), stream)
    want = oracle.embbag_bwd_dedup(ids, off, 1, dY, V, wso)
    assert got["status"] == 0 and ("resident_sort" in names) == resident
    for k in ("worker_uniq_offsets", "uniq_ids", "seg_offsets", "sorted_occ"):
        assert np.array_equal(got[k], want[k]), k
    G.close(got["uniq_grads"], want["uniq_grads"], atol=3e-6)


def test_merge_of_many_workers(stream):
    rng = np.random.default_rng(1)
    K, V, D = 40, 200_000, 8
    parts = [np.sort(rng.choice(V, size=12_000, replace=False)).astype(np.int32) for _ in range(K)]
    uid, wuo = np.concatenate(parts), np.arange(K + 1, dtype=np.int64) * 12_000
    g = rng.normal(size=(len(uid), D)).astype(np.float32)
    bsz = rng.integers(1, 50, size=K)
    _, names = G.kernels_of(lambda: G.gpu_aggregate(uid, wuo, g, bsz, V))
    assert "resident_merge" in names                   # where all SMs are there
    (ids, agg, n, _, code), names = _ran(lambda: G.gpu_aggregate(uid, wuo, g, bsz, V), stream)
    want_ids, want = oracle.aggregate_sparse(uid, wuo, g, bsz.astype(np.int64))
    assert code == 0 and n == len(want_ids) and np.array_equal(ids, want_ids) and "resident_merge" not in names
    G.close(agg, want)


def test_step_whose_sort_would_make_the_merge_order(stream):
    (t,), want = trainers("all_sms", 1)
    t.stream = stream
    _, names = _ran(t.run, stream)
    assert "resident_sort" not in names and "agg_range_emit" in names
    same(t, want)
