"""Performance cases of the batched scheduler simulation.

A case is one simulation job as a user of the package runs it: a cluster shape,
a tier mix, a seeded trace per replica, and the calls that take the trace to
its results.  ``kind`` names the calls of one pass:

* ``device``: the trace is in device memory; load, run to completion, the
  per-request results and the per-replica counters left on the device
  (parameter sweeps whose results feed further device code);
* ``host``: the trace is in host arrays; load, run, every result and the
  migration log back in host arrays (a single study, end to end);
* ``static``: ``sim_run_static``, the allocation-free call (plug-ins, hooks);
* ``adaptive``: ``adaptive.run``, the headroom controller between epochs of
  steps (set-up, chunked runs, statistics and table updates in one call);
* ``latency``: ``sim_latency_stats`` on a finished simulation (the per-tier
  reports of a sweep).

Every output is a whole number and is compared exactly: the simulation has no
rounding, so any correct implementation gives the same bits and there is no
64-bit float reference to compare against.
"""
import numpy as np
import torch

from paper_2608_16336_gb300 import adaptive, mtsim
from paper_2608_16336_gb300 import workloads as W

LENS = {"default": W.LEN_DEFAULT, "long": W.LEN_LONG_PROMPT}
DISTS = ("uniform", "gaussian", "geometric")


def _case(name, kind, replicas, instances, requests, *, blocks=2048, block_tokens=16, batch=64, tiers=4, tiers_min=0,
          dist="geometric", load=0.9, load_low=0.0, cv=1.0, lens="default", copy_blocks=64, log=0, drain=False,
          autoscale=False, epoch=0):
    c = dict(kind=kind, replicas=replicas, instances=instances, requests=requests, blocks=blocks,
             block_tokens=block_tokens, batch=batch, tiers=tiers, tiers_min=tiers_min or tiers, dist=dist, load=load,
             load_low=load_low or load, cv=cv, lens=lens, copy_blocks=copy_blocks, log=log, drain=drain,
             autoscale=autoscale, epoch=epoch)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one short what-if of a 4-instance cluster inside another program
        _case("static_probe", "static", 1, 4, 64, blocks=1024, tiers=2, dist="uniform", load=0.11, log=1024),
        # one lightly loaded 4-instance cluster, 2,000 requests, end to end from host arrays with its log
        _case("one_cluster", "host", 1, 4, 2000, blocks=1024, tiers=2, dist="uniform", load=0.11, log=32768),
        # a study of an odd shape (12-token blocks, batch 48, 33 instances) over a few dozen seeds, with logs
        _case("odd_study", "host", 97, 33, 1111, block_tokens=12, batch=48, tiers=6, dist="gaussian", load=0.8,
              log=4096),
        # many seeds of a 16-instance cluster: every replica resident at once, bound by the longest one
        _case("seeds_16", "device", 1024, 16, 2000, dist="enterprise", load=0.85, log=4096),
        # sweep over tier counts, tier mixes and loads on 32 instances
        _case("sweep_32", "device", 3840, 32, 1000, tiers=10, tiers_min=1, dist="mix", load=0.9, load_low=0.6, log=2048),
        # large sweep on 64 instances: several waves of replicas
        _case("sweep_64", "device", 8192, 64, 4000, dist="enterprise", load=0.9),
        # bursty arrivals, long prompts, many tiers on 128 instances
        _case("bursty_128", "device", 256, 128, 6000, blocks=4096, tiers=10, dist="gaussian", load=0.95, cv=3.0,
              lens="long", copy_blocks=32, log=8192),
        # the largest cluster the interface takes: 256 instances, 16 tiers
        _case("wide_256", "device", 64, 256, 6000, tiers=16, dist="uniform", load=0.9, log=8192),
        # short of KV memory: preemption and recomputation are frequent
        _case("kv_starved", "device", 700, 8, 1500, blocks=400, tiers=3, dist="uniform", load=1.3, log=4096),
        # instances being drained while the auto-scaling signal is evaluated
        _case("drain_scale", "device", 500, 24, 1500, tiers=4, dist="enterprise", load=0.8, log=4096, drain=True,
              autoscale=True),
        # the adaptive-headroom controller: epochs of steps with statistics and new tables in between
        _case("adaptive", "adaptive", 64, 16, 1000, dist="enterprise", load=0.85, log=4096, epoch=2500),
        # per-tier latency report of a finished sweep
        _case("latency_report", "latency", 1024, 16, 5000, dist="enterprise", load=0.85),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(2.0 ** rng.uniform(np.log2(lo), np.log2(hi + 0.49))))))


def draw(rng):
    kind = rng.choice(("device", "device", "device", "host", "static", "adaptive", "latency"))
    n = _log_int(rng, 1, 256)
    lens = rng.choice(("default", "default", "long"))
    bt = rng.choice((8, 12, 16, 16, 16, 32))
    blocks = max(_log_int(rng, 400, 4096), -(-(10240 if lens == "long" else 6144) // bt))
    batch = rng.choice((16, 48, 64, 64))
    tiers = rng.randint(1, 16)
    requests = _log_int(rng, 50, 1500 if kind in ("adaptive", "static") else 4000)
    most = min(8192, 16_000_000 // requests, 400_000 // n)
    if kind == "host":
        most = min(most, 128)
    if kind == "adaptive":
        most = min(most, 128)
    if kind == "static":
        per = n * (67 + 14 * tiers + bt + 16 * batch) + 1200 + 16 * requests
        most = max(1, min(64, (28 << 20) // per))
    drain = rng.random() < 0.2 and kind in ("device", "host")
    return _case("", kind, _log_int(rng, 1, most), n, requests, blocks=blocks, block_tokens=bt, batch=batch, tiers=tiers,
                 tiers_min=rng.choice((1, tiers)) if kind == "device" else tiers, dist=rng.choice(DISTS + ("mix",)),
                 load=round(rng.uniform(0.5, 1.0), 3), load_low=round(rng.uniform(0.2, 0.5), 3) if rng.random() < 0.3 else 0.0,
                 cv=rng.choice((1.0, 1.0, 3.0)), lens=lens, copy_blocks=rng.choice((16, 32, 64)),
                 log=4096 if kind in ("host", "static", "adaptive") or rng.random() < 0.5 else 0, drain=drain,
                 autoscale=rng.random() < 0.15 and kind in ("device", "host", "static"), epoch=rng.randint(500, 4000))


def workload(case, seed):
    """The cluster and the seeded traces of a case."""
    lens, n, bt = LENS[case["lens"]], case["instances"], case["block_tokens"]
    ep = W.mean_clipped_lognormal(lens["prompt_mu"], lens["prompt_sigma"], lens["prompt_min"], lens["prompt_max"])
    eo = W.mean_clipped_lognormal(lens["output_mu"], lens["output_sigma"], lens["output_min"], lens["output_max"])
    full = n * W.instance_capacity(case["blocks"], bt, case["batch"], ep, eo)
    tables, tables_k, tables_h, rt, params = {}, [], [], [], []
    span = case["tiers"] - case["tiers_min"] + 1
    for i in range(case["replicas"]):
        k = case["tiers_min"] + i % span
        if k not in tables:
            tables[k] = len(tables_k)
            tables_k.append(k)
            tables_h.append(W.headroom_decay_table(case["blocks"] // 4, k))
        rt.append(tables[k])
        dist = DISTS[(i // span) % len(DISTS)] if case["dist"] == "mix" else case["dist"]
        p = W.TgParams()
        p.seed = W.mix_seed(seed, i)
        p.num_requests = case["requests"]
        p.num_tiers = k
        p.arrival_kind = W.ARRIVAL_POISSON if case["cv"] == 1.0 else W.ARRIVAL_GAMMA
        p.rate_per_s = full * (case["load"] if i % 2 == 0 else case["load_low"])
        p.gamma_cv = case["cv"]
        for key, v in lens.items():
            setattr(p, key, v)
        p.tier_probs[:k] = W.tier_probs(dist, k)
        params.append(p)
    off, arrival, plen, olen, tier = W.generate(params)
    w = W.Workload(name="case", num_instances=n, blocks_per_instance=case["blocks"], tokens_per_block=bt,
                   max_batch=case["batch"], tables_k=tables_k, tables_h=tables_h,
                   replica_table=np.asarray(rt, np.int32), migrate_blocks_per_iter=case["copy_blocks"],
                   autoscale=int(case["autoscale"]), offsets=off, arrival_us=arrival, prompt_len=plen, output_len=olen,
                   tier=tier)
    if case["drain"]:  # a tenth of the instances start draining somewhere in the trace
        rng = np.random.default_rng(seed)
        last = arrival[off[1:] - 1].astype(np.int64)
        start = (rng.random((case["replicas"], n)) * last[:, None]).astype(np.uint32)
        w.drain_start_us = np.where(rng.random((case["replicas"], n)) < 0.1, start, np.uint32(0xFFFFFFFF))
    return w


def _ints(a):
    """A record array as plain 32-bit whole numbers."""
    return np.ascontiguousarray(a).view(np.int32)


def _device_bytes(n):
    return torch.empty(n // 4, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    w = workload(case, seed)
    s = dict(case=case, w=w)
    if case["kind"] == "adaptive":
        s["slo"] = [60_000 * (k + 1) for k in range(case["tiers"])]
        return s
    if case["kind"] == "static":
        s["trace"] = [torch.from_numpy(a).cuda() for a in (w.arrival_us.view(np.int32), w.prompt_len.view(np.int16),
                                                           w.output_len.view(np.int16), w.tier)]
        s["off"] = np.ascontiguousarray(w.offsets, np.int64)
        s["cluster"] = mtsim.sim_cluster_t(w.num_replicas, w.num_instances, w.blocks_per_instance, w.tokens_per_block,
                                           w.max_batch)
        kmax = max(w.tables_k)
        s["tk"], s["th"] = np.asarray(w.tables_k, np.int32), np.zeros((len(w.tables_k), kmax), np.int32)
        for t, h in enumerate(w.tables_h):
            s["th"][t, : len(h)] = h
        s["tiers"] = mtsim.sim_tier_table_t(len(w.tables_k), kmax, s["tk"].ctypes.data, s["th"].ctypes.data,
                                            w.replica_table.ctypes.data)
        s["policy"] = mtsim.sim_policy_t(0, w.enable_migration, w.iter_base_us, w.iter_us_per_prefill_token,
                                         w.iter_us_per_decode_seq, w.migrate_blocks_per_iter, w.theta_num, w.theta_den,
                                         case["log"], w.migrate_interval_us, w.autoscale, w.scale_out_num,
                                         w.scale_in_num, w.scale_den)
        s["res"] = _device_bytes(w.total_requests * 16)
        s["st"] = _device_bytes(w.num_replicas * 72)
        s["ev"] = torch.zeros(w.num_replicas * case["log"] * 4, dtype=torch.int32, device="cuda")
        return s
    sim = s["sim"] = mtsim.Simulator(w, event_log_capacity=case["log"])
    if case["kind"] == "device":
        sim.device_trace()
        s["res"] = _device_bytes(w.total_requests * 16)
        s["st"] = _device_bytes(w.num_replicas * 72)
    if case["kind"] == "latency":
        sim.load()
        sim.run()
        s["lat"] = _device_bytes(w.num_replicas * max(w.tables_k) * 3 * 992)
    return s


def run(s):
    case, w = s["case"], s["w"]
    kind = case["kind"]
    if kind == "static":
        t = s["trace"]
        mtsim.sim_run_static(s["cluster"], s["tiers"], s["policy"], s["off"].ctypes.data, t[0].data_ptr(),
                             t[1].data_ptr(), t[2].data_ptr(), t[3].data_ptr(), s["res"].data_ptr(),
                             s["st"].data_ptr(), s["ev"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return s["res"], s["st"], s["ev"]
    if kind == "adaptive":
        res, st, events, sched = adaptive.run(w, s["slo"], epoch_steps=case["epoch"], event_log_capacity=case["log"])
        log = np.zeros((w.num_replicas, case["log"], 6), np.int32)
        tables = np.zeros((w.num_replicas, 256, 1 + case["tiers"]), np.int32)  # the changes: step, new table
        for r in range(w.num_replicas):
            log[r, : len(events[r])] = events[r]
            for j, (step, h) in enumerate(sched[r][:256]):
                tables[r, j] = [step] + h
        return _ints(res), _ints(st), log, tables
    sim = s["sim"]
    if kind == "latency":
        mtsim.sim_latency_stats(sim.handle, s["lat"].data_ptr(), 1)
        return s["lat"]
    sim.load(on_device=kind == "device")
    sim.run()
    if kind == "device":
        mtsim.sim_metrics(sim.handle, s["res"].data_ptr(), s["st"].data_ptr(), None, 1)
        return s["res"], s["st"]
    res, st, ev = sim.metrics()
    log = _ints(ev).reshape(w.num_replicas, case["log"], 4)
    log[np.arange(case["log"]) >= st["log_events"][:, None]] = 0  # nothing was written there
    return _ints(res), _ints(st), log


def work(case):
    """Each trace record (9 bytes) and table read once, each result (16 bytes)
    and counter record (72 bytes) written once; the migration log's length is
    known only after the run and is left out.  A latency report reads the
    result and the trace fields it needs (23 bytes) and writes 992 bytes per
    replica, tier and measure.  There is no floating-point work."""
    r, q = case["replicas"], case["requests"]
    if case["kind"] == "latency":
        return {"bytes": r * q * 23 + r * case["tiers"] * 3 * 992, "flops": 0}
    return {"bytes": r * q * (9 + 16) + r * 72, "flops": 0}


def tolerance(case):
    """Whole numbers throughout: the same bits."""
    return "exact"
