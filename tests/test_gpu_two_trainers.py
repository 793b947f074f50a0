"""Several trainers on one device, each on its own stream: a step does not wait for another stream's step,
plain steps go on while another stream is being captured, and more streams than the library has side
streams for still give the same results."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200 import synth
from paper_2404_09679_b200.step import DeviceStep, OptConfig, StepBuffers
from tests.step_harness import make_batch, plan_steps

pytestmark = pytest.mark.gpu

# batches for the sort in one cluster and for the one with a CTA per SM (with a dense part on a side stream)
WORKLOADS = {"cluster": synth.WORKLOADS[1],
             "all_sms": synth.WORKLOADS[1].scaled(B=8192, dense_n=1 << 19)}


class Trainer:
    def __init__(self, w, batch, table0):
        self.w, self.b = w, batch
        nnz, n_bags = batch["row_ids"].numel(), batch["bag_offsets"].numel() - 1
        self.table, self.s0 = table0.clone(), torch.zeros_like(table0)
        self.buf = StepBuffers(w.D, w.K, nnz, n_bags, w.dense_n)
        self.step = DeviceStep(self.buf, self.table, self.s0, None, OptConfig(B.OPT_ADAGRAD, 0.01), w.K, fuse_update=True)
        self.stream = torch.cuda.Stream()

    def run(self):
        b = self.b
        self.step.run(1, b["row_ids"], b["bag_offsets"], self.w.F, b["d_pooled"], b["wso"].tolist(),
                      b["counts"].tolist(), b["dense"], stream=self.stream)

    def outputs(self):
        u = self.buf
        na = int(u.n_agg.item())
        return [u.pooled, u.agg_ids[:na], u.worker_uniq_offsets, self.table, self.s0] + \
            ([u.dense_out] if u.dense_out is not None else [])


def trainers(name, n):
    w = WORKLOADS[name]
    bm = synth.BatchMaker(w, "cuda")
    batch = make_batch(bm, plan_steps(w, 1)[0], 0)
    table0 = bm.table()
    ts = [Trainer(w, batch, table0) for _ in range(n + 1)]
    ts[-1].run()                       # alone: what every trainer must get
    torch.cuda.synchronize()
    assert B.antdt_read_status(ts[-1].buf.status) == 0
    want = [t.clone() for t in ts[-1].outputs()]
    return ts[:-1], want


def same(t, want):
    assert B.antdt_read_status(t.buf.status) == 0
    for x, y in zip(t.outputs(), want):
        assert torch.equal(x, y)


def independent(name):
    (a, b), want = trainers(name, 2)
    for t in (a, b):                   # everything loaded and created
        t.run()
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(a.stream):
        torch.cuda._sleep(1_000_000_000)
    a.run()
    done.record(a.stream)
    b.run()
    b.stream.synchronize()
    assert not done.query(), "the second trainer's step waited for the first one's"
    torch.cuda.synchronize()


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_a_step_does_not_wait_for_another_streams_step(name):
    # a process of its own: streams share hardware queues unless the driver is told otherwise at start
    r = subprocess.run([sys.executable, "-c", f"from tests.test_gpu_two_trainers import independent; independent({name!r})"],
                       env=dict(os.environ, CUDA_DEVICE_MAX_CONNECTIONS="32"), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_plain_steps_while_another_stream_is_captured(name):
    (a, b), want = trainers(name, 2)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a.stream, capture_error_mode="thread_local"):
        a.run()
        b.run()
    torch.cuda.synchronize()
    same(b, want)
    g.replay()
    torch.cuda.synchronize()
    same(a, want)


@pytest.mark.parametrize("name", list(WORKLOADS))
def test_more_streams_than_side_streams(name):
    ts, want = trainers(name, 12)
    for t in ts:
        with torch.cuda.stream(t.stream):
            torch.cuda._sleep(20_000_000)
    for t in ts:
        t.run()
    torch.cuda.synchronize()
    for t in ts:
        same(t, want)
