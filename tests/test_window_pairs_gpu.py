"""Windows with migrating pairs, bit-exact against the oracle: constant
iteration times (both ends of a pair end together), idle destinations woken
by a commit or an abort, and copies of one block per stage, at the edges of
the instances-per-lane variants."""
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


@pytest.mark.parametrize("b_us", [0, 7])  # 0: every iteration takes `base`, so times collide
@pytest.mark.parametrize("n,bmax", [(2, 4), (32, 64), (33, 16), (64, 64), (65, 8), (129, 8)])
def test_pairs(n, bmax, b_us):
    rng = np.random.default_rng(1000 * n + b_us)
    traces = []
    for gap in (5, 40, 400):  # crowded, busy and mostly idle clusters
        q = 40 + 6 * n
        a = np.cumsum(rng.integers(0, 2 * gap * 64 // n + 2, q)).astype(np.uint32)
        traces.append((a, rng.integers(1, 120, q).astype(np.uint16), rng.integers(1, 60, q).astype(np.uint16),
                       rng.integers(0, 3, q).astype(np.uint8)))
    w = W.custom(n, 60, [3], [[15, 7, 3]], [0] * len(traces), traces, tokens_per_block=4, max_batch=bmax,
                 iter_base_us=100, iter_us_per_prefill_token=0, iter_us_per_decode_seq=b_us,
                 migrate_blocks_per_iter=1 + 3 * (b_us > 0), migrate_interval_us=130, theta_num=1, theta_den=10)
    _, st, _ = parity.check_parity(w, event_log_capacity=1 << 15)
    assert int(st["migration_starts"].sum()) > 0
