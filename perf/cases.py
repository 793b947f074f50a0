"""Workloads that the framework's speed is measured on.

A case is one call pattern of a user's program at one size: whole BSP steps (through one CUDA
graph, plain launches, the four separate calls, or from host buffers), the forward alone, the
backward alone, and the server side alone.  `listed` covers the smallest calls, the ordinary ones
and the largest; `draw` gives more of the same ranges.

Keys of a case
  kind      "step" | "forward" | "backward" | "server"
  launch    steps: "graph" and "stream" (DeviceStep), "calls" (run_step's four calls), "host"
            (HostStep, two staging sets in turn)
  workers, batch, fields, rows, dim, bf16       sizes; `rows` are the table's
  bag       "fixed" | "uniform" | "poisson" with len_lo, len_hi, len_mean; shared: one hashed table
  zipf      exponent of the id distribution
  opt       "adagrad" | "adam" | "rowwise_adagrad";  fused: server step in one pass
  dense     elements of every worker's dense gradient (0: no dense part)
  dropped   server: workers whose push is disregarded (Backup Workers)
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2404_09679_b200 import binding as B
from paper_2404_09679_b200 import synth
from paper_2404_09679_b200.step import DeviceStep, HostStaging, HostStep, OptConfig, StepBuffers, run_step

_BASE = dict(kind="step", launch="stream", workers=4, batch=512, fields=8, rows=80_000, dim=16, bf16=False,
             bag="uniform", len_lo=1, len_hi=4, len_mean=0.0, shared=True, zipf=1.1, opt="adagrad",
             fused=True, dense=0, dropped=0)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest step: the tiny CPU-checkable configuration, replayed as one CUDA graph
        _case("tiny_step_graph", launch="graph", shared=False),
        # the smallest step a first user writes: the four calls one by one, odd sizes, aggregated
        # gradients kept in memory
        _case("tiny_step_calls", launch="calls", workers=5, batch=777, fields=7, rows=30_011, dim=20,
              len_hi=6, fused=False),
        # one-hot click-through step: 26 fields with a table each, one id per field, uneven workers
        _case("onehot_step_graph", launch="graph", workers=8, batch=16_384, fields=26, rows=26_000_000,
              dim=32, bag="fixed", len_hi=1, shared=False, zipf=1.05),
        # the same batch arriving in page-locked host memory every step, results read back
        _case("onehot_step_host", launch="host", workers=8, batch=16_384, fields=26, rows=26_000_000,
              dim=32, bag="fixed", len_hi=1, shared=False, zipf=1.05),
        # a cluster of many workers with small shares of the batch, one accumulator per row
        _case("many_workers_step", launch="calls", workers=90, batch=30_720, fields=39, rows=5_000_000,
              dim=16, len_hi=3, opt="rowwise_adagrad", fused=False),
        # multi-hot step, Adam, dense gradients beside the sparse ones
        _case("multihot_step_adam", workers=16, batch=65_536, fields=100, rows=10_000_000, dim=64,
              bag="poisson", len_hi=50, len_mean=10.0, opt="adam", dense=4_194_304),
        # hot-row stress: long bags over a bf16 table, heavy duplication; the largest step
        _case("hotrow_step_bf16", launch="graph", workers=16, batch=131_072, fields=40, rows=20_000_000,
              dim=64, bf16=True, bag="poisson", len_hi=100, len_mean=20.0, zipf=1.2),
        # straggler sweep: batch sizes redrawn every step, short bags, large dense part
        _case("straggler_step_adam", workers=32, batch=262_144, fields=30, rows=50_000_000, dim=32,
              len_hi=8, zipf=1.05, opt="adam", dense=16_777_216),
        # scoring requests: the forward of a handful of samples, where latency is everything
        _case("forward_request", kind="forward", batch=48, fields=26, rows=2_000_000, dim=64, bf16=True,
              len_hi=5),
        # offline evaluation: the forward of a large ragged batch with wide rows
        _case("forward_eval", kind="forward", batch=9_973, fields=31, rows=10_000_000, dim=128,
              bag="poisson", len_hi=50, len_mean=10.0),
        # one worker's backward and dedup of a mid-sized local batch, wide rows, no aggregation
        _case("backward_worker", kind="backward", workers=1, batch=6_151, fields=40, rows=1_000_003,
              dim=96, len_hi=9),
        # server side alone with two of sixteen pushes disregarded: aggregate, then the updates
        _case("backup_server_adam", kind="server", workers=16, batch=32_768, fields=50, rows=20_000_000,
              dim=64, len_hi=4, opt="adam", fused=False, dense=2_097_152, dropped=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "forward", "backward", "server"])
    dim = rng.choice([8, 16, 20, 24, 32, 40, 48, 64, 96, 128])
    bf16 = kind != "backward" and dim % 8 == 0 and rng.random() < 0.3
    bag, hi, mean = rng.choice([("fixed", 1, 1.0), ("uniform", _log_int(rng, 2, 16), 0.0),
                                ("poisson", 100, rng.uniform(3.0, 20.0))])
    avg = mean or (1 + hi) / 2
    fields = _log_int(rng, 1, 100)
    rows = max(fields, min(_log_int(rng, 10_000, 20_000_000), 640_000_000 // dim))
    most = min(60_000_000 / (fields * avg), 400_000_000 / (fields * dim))
    batch = _log_int(rng, 32, max(64.0, min(262_144.0, most)))
    workers = rng.choice([1, _log_int(rng, 2, 32), _log_int(rng, 2, 32), _log_int(rng, 33, 100)])
    workers = max(1, min(workers, batch // 8))
    opt = rng.choice(["adagrad", "adagrad", "adam"])
    launch = rng.choice(["graph", "stream", "stream", "calls", "host"]) if kind == "step" else "calls"
    if launch == "host":  # page-locked memory is dear: host batches stay below 128 MB of gradients
        batch = max(workers, min(batch, 32_000_000 // (fields * dim), int(8_000_000 / (fields * avg))))
    fused = launch != "calls" and workers <= 32 and rng.random() < 0.8
    if launch == "calls":
        opt, fused = rng.choice(["adagrad", "adam", "rowwise_adagrad"]), False
    dense = 0
    if kind in ("step", "server") and rng.random() < 0.4:
        dense = 4 * _log_int(rng, 256, max(512, 60_000_000 // workers))
        if launch == "host":
            dense = min(dense, 4_000_000 // workers * 4)
    dropped = rng.randrange(0, 3) if kind == "server" and workers > 4 else 0
    return _case(kind=kind, launch=launch, workers=workers, batch=batch, fields=fields, rows=rows, dim=dim,
                 bf16=bf16, bag=bag, len_lo=1, len_hi=hi, len_mean=mean, shared=rng.random() < 0.7,
                 zipf=round(rng.uniform(1.05, 1.2), 3), opt=opt, fused=fused, dense=dense, dropped=dropped)


# ---- inputs ---------------------------------------------------------------------------------
_stream = None


def _training_stream():
    """The stream a trainer runs on (torch's default one cannot be captured into a graph)."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


class _Zipf:
    """P(r) ~ r^-s on 1..n: the first ranks from their exact distribution, the rest from the
    continuous one (no long floating-point scan on the GPU, whose rounding changes from run to run)."""

    def __init__(self, n, s):
        m = min(n, 4096)
        w = np.arange(1, m + 1, dtype=np.float64) ** -s
        self.e, self.n = 1.0 - s, n
        self.lo, self.hi = (m + 0.5) ** self.e, (n + 0.5) ** self.e
        total = w.sum() + (self.hi - self.lo) / self.e
        self.cdf = torch.from_numpy(np.cumsum(w) / total).cuda()
        self.head = float(np.cumsum(w)[-1] / total)

    def rank(self, u):
        t = ((u - self.head) / max(1.0 - self.head, 1e-12)).clamp_(0.0, 1.0)
        tail = (self.lo + t * (self.hi - self.lo)).pow_(1.0 / self.e).round_().to(torch.int64)
        near = torch.searchsorted(self.cdf, u, right=True) + 1
        return torch.where(u < self.head, near, tail).clamp_(1, self.n)


def _bags(c, seed):
    """(row ids, bag offsets): bag lengths and field-wise Zipf ids as the synthetic workloads have
    them; a shared table gets every field's ranks hashed into it."""
    S, F = c["batch"], c["fields"]
    i64 = dict(dtype=torch.int64, device="cuda")
    smp, fld = torch.arange(S, **i64)[:, None], torch.arange(F, **i64)[None, :]
    sampler = synth.LengthSampler(c["bag"], c["len_lo"], c["len_hi"], c["len_mean"], torch.device("cuda"))
    lens = sampler.sample(synth.hash_coords(seed, synth.TAG_LEN, smp, fld)).reshape(-1)
    off = torch.zeros(S * F + 1, **i64)
    torch.cumsum(lens, 0, out=off[1:])
    nnz = int(off[-1])
    bag = torch.repeat_interleave(torch.arange(S * F, **i64), lens, output_size=nnz)
    h = synth.hash_coords(seed, synth.TAG_ID, bag, torch.arange(nnz, **i64) - off[bag])
    fld = bag % F
    per = c["rows"] if c["shared"] else c["rows"] // F
    rank = _Zipf(per, c["zipf"]).rank(synth.uniform01(h))
    if c["shared"]:
        rows = (synth.hash_coords(seed, synth.TAG_ROW, fld, rank) >> 1 & (1 << 63) - 1) % c["rows"]
    else:
        rows = fld * per + (rank - 1)
    return rows.to(torch.int32), off


def _normal(shape, std, gen, dtype=torch.float32):
    t = torch.empty(shape, dtype=dtype, device="cuda")
    return t.normal_(0.0, std, generator=gen)


def _optimizer(c, V, gen):
    """(state0, state1, OptConfig) of a run that has been going for a while: accumulators of the
    size that past mean gradients leave behind (an element seen once has |g| about 1/batch)."""
    g = 1.0 / c["batch"]
    per_row = c["opt"] == "rowwise_adagrad"
    shape = (V,) if per_row else (V, c["dim"])
    past = torch.empty(shape, device="cuda").uniform_(g * g, 4 * g * g, generator=gen)
    if c["opt"] == "adam":
        return _normal(shape, 0.3 * g, gen), past, OptConfig(B.OPT_ADAM, 1e-3, 1e-8, 0.9, 0.999)
    return past, None, OptConfig(B.OPTS[c["opt"]], 0.01, 1e-8)


def _capacity(c):
    """Occurrences and (worker, row) pairs that a program allocates for once, whatever the batch:
    the expected counts and a margin; the workers' gradients take the pairs' count only where one
    row per occurrence would be half a gigabyte or more."""
    bags, avg = c["batch"] * c["fields"], _mean_len(c)
    spread = avg if c["bag"] == "poisson" else (c["len_hi"] ** 2 - 1) / 12
    most_nnz = int(bags * avg + 6 * math.sqrt(bags * spread)) + 64
    if most_nnz * c["dim"] * 4 <= 1 << 29:
        return most_nnz, most_nnz
    return most_nnz, int(1.05 * _pairs(c)) + 1024


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    ids, off = _bags(c, seed)
    n_bags, K, D, V = off.numel() - 1, c["workers"], c["dim"], c["rows"]
    dt = torch.bfloat16 if c["bf16"] else torch.float32
    s = dict(case=c, ids=ids, off=off, status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if c["kind"] == "forward":
        s["table"] = _normal((V, D), 0.01, gen, dt)
        s["pooled"] = torch.zeros(n_bags, D, device="cuda")
        return s
    # local batches proportional to the workers' speeds, as the planner assigns them
    speeds = np.exp(0.4 * np.random.RandomState(seed % (1 << 31)).standard_normal(K)).tolist()
    s["counts"] = B.antdt_batch_sizes(speeds, K, c["batch"], B.RULE_PROPORTIONAL, 1)
    s["wso"] = [0] + [int(x) for x in np.cumsum(s["counts"])]
    s["dY"] = dY = _normal((n_bags, D), 1.0, gen)
    most_nnz, cap = _capacity(c)
    s["buf"] = buf = StepBuffers(D, K, most_nnz, n_bags, c["dense"], uniq_cap=cap, agg_cap=cap)
    for t in (buf.pooled, buf.uniq_ids, buf.seg_offsets, buf.sorted_occ, buf.uniq_grads, buf.agg_ids,
              buf.agg_grads, buf.dense_out):
        if t is not None:
            t.zero_()
    if c["kind"] == "backward":
        return s
    s["table"] = _normal((V, D), 0.01, gen, dt)
    s["s0"], s["s1"], s["oc"] = _optimizer(c, V, gen)
    s["dense"] = _normal((K, c["dense"]), 1e-2, gen) if c["dense"] else None
    if c["kind"] == "server":
        _backward(s)  # the workers' pushes that the server has in hand
        s["drop"] = [i % 5 == 2 and i // 5 < c["dropped"] for i in range(K)]
        if c["dense"]:
            s["params"] = _normal((c["dense"],), 0.01, gen)
            s["p0"] = torch.empty(c["dense"], device="cuda").uniform_(1e-6, 1e-5, generator=gen)
            s["p1"] = torch.empty(c["dense"], device="cuda").uniform_(1e-6, 1e-5, generator=gen)
    elif c["launch"] == "host":
        pin = lambda t: None if t is None else t.cpu().pin_memory()  # noqa: E731
        s["host"] = dict(ids=pin(ids), off=pin(off), dY=pin(dY), dense=pin(s["dense"]))
        s["sets"] = [HostStaging(D, K, most_nnz, n_bags, c["dense"]) for _ in range(2)]
        s["turn"] = 0
        s["step"] = HostStep(buf, s["table"], s["s0"], s["s1"], s["oc"], K, c["fused"])
    elif c["launch"] != "calls":
        s["step"] = DeviceStep(buf, s["table"], s["s0"], s["s1"], s["oc"], K, c["fused"])
    return s


# ---- one pass -------------------------------------------------------------------------------
_STEP = 100  # the global step number that the optimizers are told


def _backward(s):
    c, b = s["case"], s["buf"]
    B.antdt_embbag_bwd_dedup(s["ids"], s["off"], c["fields"], s["dY"], c["rows"], s["wso"], b.uniq_ids,
                             b.worker_uniq_offsets, b.seg_offsets, b.sorted_occ, b.uniq_grads, b.ws, b.status)


def _run_server(s):
    c, b, oc = s["case"], s["buf"], s["oc"]
    B.antdt_weighted_aggregate(s["counts"], b.ws, n_rows=c["rows"], uniq_ids=b.uniq_ids,
                               worker_uniq_offsets=b.worker_uniq_offsets, uniq_grads=b.uniq_grads,
                               agg_ids=b.agg_ids, agg_grads=b.agg_grads, n_agg=b.n_agg,
                               dense_grads=s["dense"], dense_out=b.dense_out, dev_status=b.status,
                               dropped=s["drop"] if c["dropped"] else None)
    B.antdt_sparse_opt_update(s["table"], b.agg_ids, b.agg_grads, b.n_agg, oc.opt, oc.lr, oc.eps, oc.beta1,
                              oc.beta2, _STEP, s["s0"], s["s1"], b.status)
    out = dict(agg_ids=b.agg_ids, agg_grads=b.agg_grads, n_agg=b.n_agg, table=s["table"], s0=s["s0"],
               s1=s["s1"], status=b.status)
    if c["dense"]:
        adam = oc.opt == B.OPT_ADAM
        B.antdt_dense_opt_update(s["params"], b.dense_out, B.OPT_ADAM if adam else B.OPT_ADAGRAD, oc.lr, oc.eps,
                                 oc.beta1, oc.beta2, _STEP, s["p0"], s["p1"] if adam else None)
        out.update(dense_out=b.dense_out, params=s["params"], p0=s["p0"], p1=s["p1"])
    return out


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "forward":
        B.antdt_embbag_fwd(s["table"], s["ids"], s["off"], s["pooled"], s["status"])
        return dict(pooled=s["pooled"], status=s["status"])
    b = s["buf"]
    bwd = dict(uniq_ids=b.uniq_ids, worker_uniq_offsets=b.worker_uniq_offsets, seg_offsets=b.seg_offsets,
               sorted_occ=b.sorted_occ, uniq_grads=b.uniq_grads)
    if c["kind"] == "backward":
        _backward(s)
        return dict(bwd, status=b.status)
    if c["kind"] == "server":
        return _run_server(s)
    model = dict(bwd, agg_ids=b.agg_ids, table=s["table"], s0=s["s0"], s1=s["s1"])
    if not c["fused"]:
        model["agg_grads"] = b.agg_grads
    if c["launch"] == "host":
        st, h = s["sets"][s["turn"]], s["host"]
        s["turn"] ^= 1
        st.done.synchronize()  # the step that used this set last is over
        s["step"].run(st, _STEP, h["ids"], h["off"], c["fields"], h["dY"], s["wso"], s["counts"], h["dense"],
                      stream=_training_stream(), staging_idle=True)
        return dict(model, pooled=st.h_pooled, dense_out=st.h_dense_out, n_agg=st.h_n_agg, status=st.h_status)
    if c["launch"] == "calls":
        run_step(b, s["table"], s["s0"], s["s1"], s["oc"], _STEP, s["ids"], s["off"], c["fields"], s["dY"],
                 s["wso"], s["counts"], s["dense"])
    else:
        s["step"].run(_STEP, s["ids"], s["off"], c["fields"], s["dY"], s["wso"], s["counts"], s["dense"],
                      stream=_training_stream(), graph=c["launch"] == "graph")
    return dict(model, pooled=b.pooled, n_agg=b.n_agg, dense_out=b.dense_out, status=b.status)


# ---- what a pass cannot do without ------------------------------------------------------------
def _distinct(draws, ranks, s):
    """Expected distinct values among `draws` Zipf(s) draws from 1..ranks (ranks summed in
    logarithmic buckets)."""
    edge = np.unique(np.floor(np.geomspace(1, ranks + 1, 4000)).astype(np.int64)).astype(np.float64)
    n, mid = np.diff(edge), np.sqrt(edge[:-1] * np.maximum(edge[1:] - 1, edge[:-1]))
    p = mid ** -s
    p /= np.sum(n * p)
    return float(np.sum(n * -np.expm1(draws * np.log1p(-np.minimum(p, 1 - 1e-12)))))


def _mean_len(c):
    return c["len_mean"] if c["bag"] == "poisson" else (c["len_lo"] + c["len_hi"]) / 2


def _pairs(c, workers=None):
    """Expected distinct (worker, row) pairs of a batch; workers=1: distinct rows."""
    K = workers or c["workers"]
    draws = c["batch"] * _mean_len(c) / K
    ranks = c["rows"] if c["shared"] else max(1, c["rows"] // c["fields"])
    return min(K * c["rows"], K * c["fields"] * min(draws, _distinct(draws, ranks, c["zipf"])))


def work(case):
    c = case
    D, K, F, S = c["dim"], c["workers"], c["fields"], c["batch"]
    bags, nnz, ew = S * F, S * F * _mean_len(c), 2 if c["bf16"] else 4
    u, su = _pairs(c, 1), _pairs(c)
    csr = 4 * nnz + 8 * (bags + 1)
    forward = u * D * ew + 4 * bags * D
    backward = 4 * bags * D + 4 * nnz + su * (4 + 8 + 4 * D)
    state = {"adagrad": 8 * D, "adam": 16 * D, "rowwise_adagrad": 8}[c["opt"]]
    update = u * (4 + 2 * D * ew + state)
    dense = 4 * c["dense"] * (K + 1)
    if c["kind"] == "forward":
        return {"bytes": csr + forward, "flops": nnz * D}
    if c["kind"] == "backward":
        return {"bytes": csr + backward, "flops": nnz * D}
    kept = (K - c["dropped"]) / K
    if c["kind"] == "server":
        tuned = 4 * c["dense"] * (6 if c["opt"] == "adam" else 4)
        return {"bytes": kept * su * (4 + 4 * D) + 4 * u * D + update + kept * dense + tuned,
                "flops": 2 * su * D + 8 * u * D + 2 * c["dense"] * K}
    host = 0.0
    if c["launch"] == "host":  # every input enters and every result leaves through the host link once
        host = csr + 8 * bags * D + dense
    kept_grads = 0 if c["fused"] else 4 * u * D
    return {"bytes": csr + forward + backward + update + dense + kept_grads + host,
            "flops": 2 * nnz * D + 2 * su * D + 8 * u * D + 2 * c["dense"] * K}


def tolerance(case):
    # fp32 sums in another order; bf16 rows can land on the neighbouring value
    return {"rel": 2e-4, "max": 0.02} if case["bf16"] and case["kind"] != "forward" else {"rel": 1e-5, "max": 5e-4}
