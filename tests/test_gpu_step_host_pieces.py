"""antdt_bsp_step_host with a d_pooled large enough to travel in several pieces: every output must equal
the device-resident step's bit for bit, with even workers, one dominant worker and empty ones."""
import pytest
import torch

from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200 import synth
from paper_2404_09679_b200.step import DeviceStep, HostStaging, HostStep, OptConfig, StepBuffers
from tests.step_harness import make_batch, plan_steps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [[16_384] * 4, [64_000, 0, 0, 1536], [0, 20_000, 45_536, 0]])
def test_host_step_in_pieces_equals_the_device_step(counts):
    w = synth.WORKLOADS[3].scaled(K=4, B=65_536, F=48, V=300_000, dense_n=0, len_mean=3.0, speed_kind="equal")
    assert w.B * w.F * w.D * 4 >= 3 << 28       # three pieces of 256 MB or more
    b = make_batch(synth.BatchMaker(w, "cuda"), plan_steps(w, 1)[0], 0)
    wso = [sum(counts[:i]) for i in range(5)]
    nnz, n_bags = b["row_ids"].numel(), b["bag_offsets"].numel() - 1
    table0 = torch.randn(w.V, w.D, device="cuda", generator=torch.Generator("cuda").manual_seed(1)) * 0.01
    oc = OptConfig(B.OPT_ADAGRAD, 0.01)
    out = []
    for host in (False, True):
        table, s0 = table0.clone(), torch.zeros(w.V, w.D, device="cuda")
        buf = StepBuffers(w.D, 4, nnz, n_bags)
        if host:
            st, step = HostStaging(w.D, 4, nnz, n_bags), HostStep(buf, table, s0, None, oc, 4)
            pin = [b[k].cpu().pin_memory() for k in ("row_ids", "bag_offsets", "d_pooled")]
            step.run(st, 1, pin[0], pin[1], w.F, pin[2], wso, counts)
            st.done.synchronize()
            assert int(st.h_status[0]) == 0
            pooled = st.h_pooled.cuda()
        else:
            DeviceStep(buf, table, s0, None, oc, 4).run(1, b["row_ids"], b["bag_offsets"], w.F, b["d_pooled"], wso,
                                                        counts)
            assert B.antdt_read_status(buf.status) == 0
            pooled = buf.pooled
        nu = int(buf.worker_uniq_offsets[4].item())
        out.append((pooled[:n_bags].clone(), buf.uniq_ids[:nu].clone(), buf.uniq_grads[:nu].clone(), table, s0))
    for x, y in zip(*out):
        assert torch.equal(x, y)
