"""The forward's call from Python (csrc/marshal.cpp): what it takes directly, and what goes the general way and is
refused there as before; and the library without that module."""
import sys
import types

import numpy as np
import pytest
import torch

from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200 import build


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


@pytest.fixture(params=["absent", "of another torch", "without a version"])
def no_module(request, monkeypatch):
    mod = None                                               # the import system's mark of a module that is not there
    if request.param != "absent":
        mod = types.ModuleType("_marshal")
        mod.bind = mod.embbag_fwd = lambda *_: pytest.fail("used")
        if request.param == "of another torch":
            mod.torch_version = "0.0"
    pkg = sys.modules["paper_2404_09679_b200"]
    monkeypatch.delattr(pkg, "_marshal", raising=False)
    monkeypatch.setitem(sys.modules, "paper_2404_09679_b200._marshal", mod)
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "_fwd", None)


def test_the_library_does_without_the_module(no_module):
    assert list(B.antdt_batch_sizes([1.0] * 4, 4, 8)) == [2, 2, 2, 2]
    ids, off = torch.zeros(3, dtype=torch.int32), torch.tensor([0, 3])
    table, pooled = torch.zeros(4, 8), torch.zeros(1, 8)
    assert B._fwd(table, ids, off, pooled, None, None) == -1
    with pytest.raises(AssertionError):
        B.antdt_embbag_fwd(table.t(), ids, off, pooled)
    with pytest.raises(B.AntdtError):
        B.antdt_embbag_fwd(table.half(), ids, off, pooled)


def test_a_module_of_another_torch_or_python_is_built_again(monkeypatch, tmp_path):
    monkeypatch.setattr(build, "MARSHAL", str(tmp_path / "m.so"))
    monkeypatch.setattr(build, "MARSHAL_KEY", str(tmp_path / "key"))
    assert not build._marshal_current(0.0)
    (tmp_path / "m.so").write_bytes(b"")
    assert not build._marshal_current(0.0)
    (tmp_path / "key").write_text(build._marshal_key())
    assert build._marshal_current(0.0) and not build._marshal_current(1e12)
    monkeypatch.setattr(torch, "__version__", "0.0")
    assert not build._marshal_current(0.0)


@pytest.mark.gpu
def test_a_forward_without_the_module(no_module):
    test_streams_status_and_subclasses()
    assert B._fwd is B._general_only


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
