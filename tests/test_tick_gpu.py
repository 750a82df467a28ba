"""The rebalancing tick at the edges of its ranking and of its loop choice,
bit-exact against the oracle: instance counts around the four-key steps of
the ranking and around 32 pairs, theta = 0 (the pair-by-pair search) and
theta > 0, destinations without room (a source's candidate does not fit), and
replica counts on both sides of the choice between the two main loops."""
import numpy as np
import pytest

from paper_2608_16336_gb300 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


def _trace(rng, n, q, k, long_prompts):
    a = np.cumsum(rng.integers(0, max(2, 600 // n), q)).astype(np.uint32)
    p = rng.integers(1, 300 if long_prompts else 40, q)
    return a, p.astype(np.uint16), rng.integers(1, 60, q).astype(np.uint16), rng.integers(0, k, q).astype(np.uint8)


@pytest.mark.parametrize("theta", [(0, 1), (1, 1000), (3, 10)])
@pytest.mark.parametrize("n", [2, 3, 31, 32, 63, 64, 66, 127, 256])
def test_tick(n, theta):
    rng = np.random.default_rng(n)
    traces = [_trace(rng, n, 60 + 5 * n, 3, lp) for lp in (False, True)]
    w = W.custom(n, 100, [3], [[20, 10, 5]], [0, 0], traces, tokens_per_block=4, max_batch=64, iter_base_us=200,
                 iter_us_per_prefill_token=1, iter_us_per_decode_seq=3, migrate_blocks_per_iter=8,
                 migrate_interval_us=350, theta_num=theta[0], theta_den=theta[1])
    _, st, _ = parity.check_parity(w, event_log_capacity=1 << 16)
    assert int(st["log_events"].sum()) > 0


@pytest.mark.parametrize("n,replicas", [(30, 1519), (30, 1521), (40, 2127), (40, 2129), (40, 3951), (40, 3953), (8, 1519),
                                        (8, 1521), (16, 1300)])
def test_both_loops(n, replicas):
    """One per lane and two per lane, records in HBM or shared, around the replica counts
    where a 152-SM GPU changes loops and scratch; sampled replicas against the oracle."""
    rng = np.random.default_rng(replicas)
    traces = [_trace(rng, n, 40, 2, r % 2 == 0) for r in range(replicas)]
    w = W.custom(n, 90, [2], [[18, 9]], [0] * replicas, traces, tokens_per_block=4, max_batch=64, iter_base_us=200,
                 iter_us_per_prefill_token=1, iter_us_per_decode_seq=3, migrate_blocks_per_iter=8,
                 migrate_interval_us=350, theta_num=3, theta_den=10)
    parity.check_parity(w, replicas=[0, 1, replicas // 2, replicas - 1], event_log_capacity=512)
