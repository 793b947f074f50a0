"""The backward on offsets that do not cover the ids, with a workspace full of old data: the error is
flagged and nothing outside the output buffers is written, whichever sort the input takes (a cluster, one
CTA per SM, the multi-kernel sort)."""
import numpy as np
import pytest
import torch

from paper_2404_09679_b200 import binding as B
from tests import gpu_util as G

pytestmark = pytest.mark.gpu
GUARD = 4096


def _guarded(shape, dtype):
    n = int(np.prod(shape))
    whole = torch.full((n + 2 * GUARD,), -7, dtype=dtype, device="cuda")
    return whole, whole[GUARD:GUARD + n].view(shape)


@pytest.mark.parametrize("fill", [0xFF, 0x7F, 0x80])
@pytest.mark.parametrize("bad", ["short", "all_zero", "late_start"])
@pytest.mark.parametrize("n_bags,K", [(1500, 3), (30_000, 3), (30_000, 129)])
def test_nothing_outside_the_outputs_is_written(n_bags, K, bad, fill):
    rng = np.random.default_rng(n_bags)
    D, V, nnz = 16, 1000, 3 * n_bags
    off = np.arange(n_bags + 1, dtype=np.int64) * 3
    if bad == "short":
        off = np.minimum(off, nnz // 3)
    elif bad == "all_zero":
        off[:] = 0
    else:
        off = np.maximum(off, nnz // 2)
    wso = np.concatenate([[0], np.sort(rng.integers(0, n_bags + 1, size=K - 1)), [n_bags]]).tolist()
    ids = G.dev(rng.integers(0, V, size=nnz).astype(np.int32))
    dY = torch.ones(n_bags, D, device="cuda")
    size = B.antdt_embbag_bwd_dedup_workspace_bytes(nnz, n_bags, D, K)
    out = dict(ug=_guarded((nnz, D), torch.float32), uid=_guarded((nnz,), torch.int32),
               so=_guarded((nnz + 1,), torch.int64), occ=_guarded((nnz,), torch.int32),
               wuo=_guarded((K + 1,), torch.int64))
    ws = torch.full((size,), fill, dtype=torch.uint8, device="cuda")
    st = G.new_status()
    B.antdt_embbag_bwd_dedup(ids, G.dev(off), 1, dY, V, wso, out["uid"][1], out["wuo"][1], out["so"][1], out["occ"][1],
                             out["ug"][1], ws, st)
    assert B.antdt_read_status(st) == B.ERR_BAD_OFFSETS
    for name, (whole, _) in out.items():
        assert (whole[:GUARD] == -7).all() and (whole[-GUARD:] == -7).all(), name
