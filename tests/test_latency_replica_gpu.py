"""Latency statistics at the edges of the one-kernel path (replicas of 0 to
16,383 requests, the block sizes it changes at, ragged warps, the tier counts
whose shared memory differs, all values alike, the largest replicas its shared
memory holds) and past it, where the streaming passes take replicas of any size
together, bit-exact against sorted values."""
import threading

import numpy as np
import pytest

from paper_2608_16336_gb300 import mtsim
from paper_2608_16336_gb300 import workloads as W
from tests.test_latency_gpu import compare, gpu_stats

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _workload(sizes, k, alike, seed):
    rng = np.random.default_rng(seed)
    traces = []
    for q in sizes:
        a = np.cumsum(rng.integers(0, 120, q)).astype(np.uint32)
        p, o = rng.integers(1, 200, q), rng.integers(1, 9, q)
        traces.append((a, p.astype(np.uint16), o.astype(np.uint16), rng.integers(0, k, q).astype(np.uint8)))
    b = 0 if alike else 5
    return W.custom(2, 4096, [k], [[64 >> i for i in range(k)]], [0] * len(sizes), traces, iter_base_us=300,
                    iter_us_per_prefill_token=b, iter_us_per_decode_seq=b)


@pytest.mark.parametrize("sizes", [(0, 1, 2, 31, 32, 33, 512), (511, 513, 0, 1024), (1025, 3, 8192), (8193, 129)])
@pytest.mark.parametrize("k", [1, 4, 5, 16])
def test_sizes(sizes, k):
    w = _workload(sizes, k, False, 7 * k + len(sizes))
    compare(w, gpu_stats(w), range(len(sizes)))


@pytest.mark.parametrize("q", [16383, 16384])
@pytest.mark.parametrize("alike", [False, True])
def test_largest(q, alike):
    w = _workload((q,), 1, alike, q)
    compare(w, gpu_stats(w), [0])


@pytest.mark.parametrize("q,k", [(8192, 4), (8191, 1), (4000, 16)])
def test_one_block_per_sm(q, k):
    """More replicas than SMs, each filling an SM's shared memory (or, with one tier, half of it)."""
    w = _workload((q,) * 160, k, False, q)
    compare(w, gpu_stats(w), [0, 80, 159])


@pytest.mark.parametrize("q,k", [(16064, 4), (16065, 4), (10608, 16), (10609, 16)])
def test_shared_memory_limit(q, k):
    """The largest replica that a block's 227 KB holds, and one request more."""
    w = _workload((q, 7), k, False, q)
    compare(w, gpu_stats(w), range(2))


@pytest.mark.parametrize("max_steps", [None, 4000])
@pytest.mark.parametrize("k", [1, 16])
def test_streaming_mixed_sizes(k, max_steps):
    """Empty and tiny replicas beside large ones, finished or stopped early, to host and device."""
    import torch
    w = _workload((0, 17000, 3, 4096, 0, 16500, 4097), k, False, 5 + k)
    sim = mtsim.Simulator(w, event_log_capacity=0)
    try:
        sim.load()
        sim.run() if max_steps is None else sim.run(max_steps)
        host = sim.latency_stats()
        d = torch.empty(host.nbytes, dtype=torch.uint8, device="cuda")
        mtsim.sim_latency_stats(sim.handle, d.data_ptr(), 1)
        torch.cuda.synchronize()
    finally:
        sim.close()
    assert d.cpu().numpy().tobytes() == host.tobytes()
    compare(w, host, range(w.num_replicas), **({} if max_steps is None else dict(max_steps=max_steps)))


def test_unfinished_requests_left_out():
    w = _workload((700, 40), 3, False, 3)
    compare(w, gpu_stats(w, max_steps=150), range(2), max_steps=150)


@pytest.mark.parametrize("sizes", [((40,), (400,)), ((17000,), (17001, 5))])  # one kernel; streaming passes
def test_two_host_threads(sizes):
    """Objects in use by two host threads whose launches take different shared memory."""
    ws = [_workload(s, k, False, 11 + k) for s, k in zip(sizes, (9, 16))]
    sims = [mtsim.Simulator(w, event_log_capacity=0) for w in ws]
    errors, got = [], [None, None]

    def work(i):
        try:
            for _ in range(3000):
                got[i] = sims[i].latency_stats()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    try:
        for s in sims:
            s.load()
            s.run()
        threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        assert not errors, errors[0]
        for w, g in zip(ws, got):
            compare(w, g, range(w.num_replicas))
    finally:
        for s in sims:
            s.close()
