"""Device steps back to back on one stream: the forward of a small step, which runs beside its sort on a side
stream, must read the table as the step before it (with a long update) leaves it."""
import pytest
import torch

from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200.step import DeviceStep, OptConfig, StepBuffers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("small", [500, 20_000, 60_000])     # one cluster, a large one, one CTA per SM
def test_forward_sees_the_update_before_it(small):
    V, D, K = 1_000_000, 64, 2
    gen = torch.Generator("cuda").manual_seed(1)
    table = torch.randn(V, D, device="cuda", generator=gen) * 0.01
    state = torch.full((V, D), 1e-4, device="cuda")
    stream = torch.cuda.Stream()

    def make(n, lr):
        ids = torch.randperm(V, device="cuda", generator=gen)[:n].to(torch.int32)
        off = torch.arange(n + 1, dtype=torch.int64, device="cuda")
        dY = torch.randn(n, D, device="cuda", generator=gen)
        buf = StepBuffers(D, K, n, n)
        step = DeviceStep(buf, table, state, None, OptConfig(B.OPT_ADAGRAD, lr), K, fuse_update=True)
        half = n // 2
        return buf, ids, lambda: step.run(1, ids, off, 1, dY, [0, half, n], [half, n - half], stream=stream)

    big, _, run_big = make(V, 0.1)
    buf, ids, run_small = make(small, 0.0)         # at rate 0 it leaves the table as it reads it
    torch.cuda.synchronize()
    for _ in range(30):
        run_big()
        run_small()
        stream.synchronize()
        assert torch.equal(buf.pooled[:small], table[ids.long()])
    assert B.antdt_read_status(buf.status) == 0 and B.antdt_read_status(big.status) == 0
