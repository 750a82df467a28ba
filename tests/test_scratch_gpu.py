"""Shared memory of the simulation kernel.  Replica counts at which a smaller per-warp scratch makes every replica
resident on 152 SMs, or would if it held less than the shape needs, with four
and eight instances per lane: ticks that rank all instances and windows in which
most of them form a batch; states that leave little room; live objects whose
kernels are the same and whose shared memory differs.  Bit-exact against the
oracle."""
import numpy as np
import pytest

from paper_2608_16336_gb300 import mtsim
from paper_2608_16336_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _workload(n, k, replicas, block_tokens=16, batch=64):
    """Constant iteration times and arrivals a microsecond or two apart: hundreds
    of instances end and form batches in the same window."""
    rng = np.random.default_rng(n + k)
    q = 3 * n
    traces = [(np.cumsum(rng.integers(0, 3, q)).astype(np.uint32), rng.integers(1, 60, q).astype(np.uint16),
               rng.integers(1, 40, q).astype(np.uint16), rng.integers(0, k, q).astype(np.uint8))
              for _ in range(replicas)]
    return W.custom(n, 100, [k], [[max(1, 20 >> i) for i in range(k)]], [0] * replicas, traces, tokens_per_block=block_tokens,
                    max_batch=batch, iter_base_us=200, iter_us_per_prefill_token=0, iter_us_per_decode_seq=0,
                    migrate_blocks_per_iter=8, migrate_interval_us=350, theta_num=1, theta_den=1000)


def shared_bytes(w):
    sim = mtsim.Simulator(w, event_log_capacity=0)
    try:
        return sim.launch_info()["shared_bytes"]
    finally:
        sim.close()


@pytest.mark.parametrize("n,k,replicas,shrunk", [(250, 4, 700, False), (196, 7, 700, False), (196, 14, 400, False),
                                                 (244, 4, 700, True), (256, 1, 1100, True), (123, 15, 700, True)])
def test_scratch_at_its_least(n, k, replicas, shrunk):
    import torch
    w = _workload(n, k, replicas)
    if torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert (shared_bytes(w) < shared_bytes(_workload(n, k, 2))) == shrunk
    _, st, _ = parity.check_parity(w, replicas=[0, 1, replicas // 2, replicas - 1], event_log_capacity=1 << 12)
    assert int(st["log_events"].sum()) > 0


@pytest.mark.parametrize("n,block_tokens,records_in_shared", [(256, 52, 1), (249, 64, 1), (254, 60, 0), (256, 64, 0)])
def test_largest_state_beside_the_records(n, block_tokens, records_in_shared):
    """16 tiers and a batch of 6: the records and a 4 KB scratch do not fit together."""
    w = _workload(n, 16, 3, block_tokens, 6)
    sim = mtsim.Simulator(w, event_log_capacity=0)
    try:
        assert sim.launch_info()["slots_in_shared"] == records_in_shared
    finally:
        sim.close()
    parity.check_parity(w, event_log_capacity=1 << 14)


@pytest.mark.parametrize("first,second", [((128, 8, 64), (128, 8, 1000)), ((128, 8, 1000), (128, 8, 64)),
                                          ((256, 16, 2), (256, 1, 3)), ((64, 16, 2), (40, 9, 2))])
def test_live_objects(first, second):
    """Neither object's launch depends on what the other planned, in either order."""
    ws = [_workload(*first), _workload(*second)]
    sims = [mtsim.Simulator(w, event_log_capacity=1 << 12) for w in ws]
    try:
        assert sims[0].launch_info()["shared_bytes"] != sims[1].launch_info()["shared_bytes"]
        for s in sims:
            s.load()
        for w, s in zip(ws, sims):
            assert s.run() == 0
            res, st, ev = s.metrics()
            events = [s.events_of(ev, st, r) for r in range(w.num_replicas)]
            ref = parity.run_oracle(w, [0, w.num_replicas - 1], event_log_capacity=1 << 12)
            for r in (0, w.num_replicas - 1):
                parity.compare_replica(w, r, res, st, events, ref[r])
    finally:
        for s in sims:
            s.close()


@pytest.mark.parametrize("n,k,replicas", [(2, 2, 1064), (2, 2, 1065), (16, 4, 1521), (32, 4, 1825), (32, 4, 2433),
                                          (40, 4, 1825), (64, 4, 2737), (64, 4, 3648), (64, 16, 2432), (100, 4, 1400), (100, 4, 2048)])
def test_loop_edges(n, k, replicas):
    """Replica counts on either side of the choice between the two main loops on 152 SMs."""
    w = _workload(n, k, replicas)
    _, st, _ = parity.check_parity(w, replicas=[0, 1, replicas // 2, replicas - 1], event_log_capacity=1 << 10)
    assert int(st["finished"].sum()) == w.total_requests
