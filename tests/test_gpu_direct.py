"""Small calls (records straight into the table) against the oracle, at the sizes where the route changes."""
import numpy as np
import pytest

import oracle
from tests.helpers import sorted_by_key
from tracegen.layout import RECORD_DTYPE

pytestmark = pytest.mark.gpu
PEAK_BW, PEAK_FLOPS = 8e12, [1e15] * 8


def trace(n, law, seed):
    rng = np.random.default_rng(seed)
    r = np.zeros(n, dtype=RECORD_DTYPE)
    r["app_id"] = rng.integers(0, 9, n)                       # one application in nine does not exist
    r["phase"] = rng.integers(0, 3, n)
    if law == "one key":
        r["phase"], r["op_id"], r["shape_id"] = 1, 7, 0xFFFFFFFF
    elif law == "few":
        r["op_id"], r["shape_id"] = rng.integers(0, 3, n), rng.integers(0, 5, n)
    else:
        r["op_id"], r["shape_id"] = rng.integers(0, 1 << 16, n), rng.integers(0, 1 << 32, n, dtype=np.uint64)
    r["duration_ns"] = rng.choice(np.array([0, 1, 50_000, 0x0FFFFFFF, 0xFFFFFFFF], dtype=np.uint32), n)
    return r


@pytest.mark.parametrize("law", ["one key", "few", "distinct"])
@pytest.mark.parametrize("n", [1, 33, 127, 129, 8_192, 8_193, 70_001, (1 << 18) + 1, 1 << 20, (1 << 20) + 1])
def test_small_calls_match_the_oracle(n, law):
    import torch
    import paper_2607_14541_b200 as p
    weights = np.array([0xFFFFFFFF, 1, 0x00100000, 0x000FFFFF, 3, 5, 7, 0], dtype=np.uint32)
    recs = trace(n, law, n)
    agg = p.Aggregator(weights, 3, max(n, 16))
    dev = torch.from_numpy(recs.view(np.uint8).reshape(-1)).cuda()
    for _ in range(2):                                        # the second call meets the first one's keys
        agg.ingest(dev, n=n)
    o = oracle.Oracle(weights, 3)
    o.ingest(np.concatenate([recs, recs]), threads=4)
    got = sorted_by_key(agg.finalize_numpy(PEAK_BW, PEAK_FLOPS))
    assert got.tobytes() == o.finalize(PEAK_BW, PEAK_FLOPS).tobytes()
    st = agg.stats()
    assert st["n_valid"] + st["n_rejected"] == 2 * n and st["n_rejected"] == 2 * int((recs["app_id"] >= 8).sum())


def test_a_first_host_call_goes_direct_whatever_its_size():
    """Into a table that stays in L2, every piece of a host call takes one direct launch (the rule looks at the records of
    earlier calls); the next device call, with more than 2^22 records before it, takes the two-pass route."""
    import torch
    import paper_2607_14541_b200 as p
    weights = np.arange(1, 9, dtype=np.uint32)
    n, later = (1 << 22) + 5, 1 << 18
    recs = trace(n + later, "few", 11)
    host = torch.from_numpy(recs[:n].view(np.uint8).reshape(-1)).pin_memory()
    agg = p.Aggregator(weights, 3, 4096)
    before = agg.launch_count()
    agg.ingest_host(host, n=n)
    assert agg.launch_count() - before == 2 and len(agg.hot_directory()) == 0
    agg.ingest(torch.from_numpy(recs[n:].view(np.uint8).reshape(-1)).cuda(), n=later)
    assert len(agg.hot_directory()) > 0
    o = oracle.Oracle(weights, 3)
    o.ingest(recs, threads=4)
    assert sorted_by_key(agg.finalize_numpy(PEAK_BW, PEAK_FLOPS)).tobytes() == o.finalize(PEAK_BW, PEAK_FLOPS).tobytes()
