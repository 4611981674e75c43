"""What the hot directory's sample makes of traces whose neighbouring records are not independent."""
import numpy as np
import pytest

from tracegen.layout import RECORD_DTYPE

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("law", ["runs", "periodic"])
def test_frequent_keys_are_found_in_traces_with_patterns(law):
    """runs: every key comes four times in a row; 4 096 keys hold an eighth of the trace, the others come once.
    periodic: 512 keys take every 32nd place, the rest is spread over 2^20.  Of 2^18 sampled records a frequent key
    has 8 (a seventieth of the keys fewer than the three that are needed) and 16; crowded buckets cost some more."""
    import torch
    import paper_2607_14541_b200 as p
    rng, n = np.random.default_rng(7), 1 << 23
    if law == "runs":
        n_hot, runs = 4096, n // 4
        key = np.repeat(np.where(rng.random(runs) < 1 / 8, rng.integers(0, n_hot, runs), n_hot + np.arange(runs)), 4)
    else:
        n_hot = 512
        key = np.where(np.arange(n) % 32 == 17, rng.integers(0, n_hot, n), n_hot + rng.integers(0, 1 << 20, n))
    recs = np.zeros(n, dtype=RECORD_DTYPE)
    recs["op_id"], recs["shape_id"], recs["duration_ns"] = key % 61, key, 1000
    agg = p.Aggregator(np.ones(1, dtype=np.uint32), 1, 1 << 21)
    agg.ingest(torch.from_numpy(recs.view(np.uint8).reshape(-1)).cuda(), n=n)
    assert agg.stats()["n_valid"] == n
    held = (agg.hot_directory() & np.uint64(0xFFFFFFFF)) < n_hot
    assert held.sum() >= 0.95 * n_hot
