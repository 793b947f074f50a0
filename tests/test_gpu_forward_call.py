"""The forward's call from Python (csrc/marshal.cpp): what it takes directly, and what goes the general way and is
refused there as before."""
import numpy as np
import pytest
import torch

from paper_2404_09679_b200 import binding as B


def test_what_is_not_a_plain_contiguous_tensor_goes_the_general_way():
    B.lib()
    ids, off = torch.zeros(3, dtype=torch.int32), torch.tensor([0, 3])
    table, pooled = torch.zeros(4, 8), torch.zeros(1, 8)

    class Sub(torch.Tensor):
        pass

    for args in [(table.t(), ids, off, pooled), (table.double(), ids, off, pooled), (table[0], ids, off, pooled),
                 (table, torch.zeros(6, dtype=torch.int32)[::2], off, pooled), (table, ids, off, pooled.as_subclass(Sub)),
                 (table, ids, off, 7)]:
        assert B._fwd(*args, None, None) == -1
    with pytest.raises(AssertionError):
        B.antdt_embbag_fwd(table.t(), ids, off, pooled)
    with pytest.raises(B.AntdtError):
        B.antdt_embbag_fwd(table.half(), ids, off, pooled)


@pytest.mark.gpu
def test_streams_status_and_subclasses():
    rng = np.random.default_rng(1)
    table = torch.nn.Parameter(torch.from_numpy(rng.normal(size=(50, 8)).astype(np.float32)).cuda())
    ids = torch.from_numpy(rng.integers(0, 50, size=64).astype(np.int32)).cuda()
    off = torch.arange(0, 65, 4, device="cuda")
    want = table.detach()[ids.long()].view(16, 4, 8).sum(1)
    side = torch.cuda.Stream()

    class Sub(torch.Tensor):
        pass

    for tab, stream in [(table, None), (table.detach(), side), (table.detach().as_subclass(Sub), None)]:
        out, st = torch.zeros(16, 8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        B.antdt_embbag_fwd(tab, ids, off, out, st, stream)
        with torch.cuda.stream(side):
            B.antdt_embbag_fwd(tab, ids, off, out)           # no status word, the current stream
        torch.cuda.synchronize()
        assert torch.allclose(out, want, rtol=1e-5, atol=1e-6) and int(st) == 0
    ids[5] = 50
    B.antdt_embbag_fwd(table, ids, off, out, st)
    assert B.antdt_read_status(st) == B.ERR_ID_OUT_OF_RANGE
    with pytest.raises(B.AntdtError) as e:                   # refused by the entry point itself
        B.antdt_embbag_fwd(torch.zeros(4, 6, device="cuda"), ids, off, out)
    assert e.value.code == B.ERR_INVALID_ARG
