"""Entries of a finalize against the oracle where the work table's buckets and the warps' batches of entries end."""
import numpy as np
import pytest

import oracle
from tests.helpers import sorted_by_key
from tracegen.layout import RECORD_DTYPE, WORK_DTYPE

pytestmark = pytest.mark.gpu
PEAK_BW, PEAK_FLOPS = 7.7e12, [1e15 * (i + 1) / 3 for i in range(8)]


def inputs(n_keys, n_rows, seed):
    """n_keys different (operator, shape), and a work table that holds two of three of them beside others."""
    rng = np.random.default_rng(seed)
    pair = rng.permutation(4 * n_keys)[: 2 * n_keys]
    recs = np.zeros(n_keys, dtype=RECORD_DTYPE)
    recs["op_id"], recs["shape_id"] = pair[:n_keys] % 97, pair[:n_keys]
    recs["phase"], recs["duration_ns"] = rng.integers(0, 2, n_keys), rng.integers(0, 1 << 32, n_keys, dtype=np.uint64)
    listed = np.concatenate([pair[:n_keys][np.arange(n_keys) % 3 != 1], pair[n_keys:]])[:n_rows]
    work = np.zeros(len(listed), dtype=WORK_DTYPE)
    work["op_id"], work["shape_id"], work["dtype"] = listed % 97, listed, rng.integers(0, 8, len(listed))
    for field in ("flops", "bytes"):
        work[field] = rng.integers(0, 1 << 64, len(listed), dtype=np.uint64) >> rng.integers(0, 64, len(listed), dtype=np.uint64)
    return recs, work


@pytest.mark.parametrize("n_rows", [0, 1, 5, 1_000, 1 << 30])
@pytest.mark.parametrize("n_keys,max_keys", [(1, 100_000), (33, 100_000), (60_001, 60_001), (300_007, 300_007), (700, 700), (20_000, 20_000)])
def test_entries_match_the_oracle(n_keys, max_keys, n_rows):
    """(up to 25 000 provisioned keys the cluster's kernel, above the one with a warp per 128 slots; the work table as small
    as its rows)"""
    import torch
    import paper_2607_14541_b200 as p
    recs, work = inputs(n_keys, n_rows, n_keys + n_rows)
    weights = np.array([7, 0], dtype=np.uint32)
    agg = p.Aggregator(weights, 2, max_keys, max_work_rows=len(work))
    o = oracle.Oracle(weights, 2)
    if len(work):
        agg.set_work_table(work)
        o.set_work(work)
    agg.ingest(torch.from_numpy(recs.view(np.uint8).reshape(-1)).cuda(), n=n_keys)
    o.ingest(recs, threads=4)
    exp = o.finalize(PEAK_BW, PEAK_FLOPS)
    out = torch.full((48 * (n_keys + 1),), 0xA5, dtype=torch.uint8, device="cuda")
    got, n = agg.finalize(PEAK_BW, PEAK_FLOPS, out=out)
    assert n == len(exp) == n_keys
    host = out.cpu().numpy()
    assert sorted_by_key(host[: 48 * n].view(p.ENTRY_DTYPE)).tobytes() == exp.tobytes()
    assert (host[48 * n:] == 0xA5).all()


@pytest.mark.parametrize("cap", [1, 31, 60_000])
def test_a_list_that_does_not_fit_is_cut_at_its_end(cap):
    import torch
    import paper_2607_14541_b200 as p
    recs, work = inputs(60_001, 1_000, 3)
    agg = p.Aggregator(np.array([7], dtype=np.uint32), 2, 60_001, max_work_rows=len(work))
    agg.set_work_table(work)
    agg.ingest(torch.from_numpy(recs.view(np.uint8).reshape(-1)).cuda(), n=len(recs))
    out = torch.full((48 * (cap + 64),), 0xA5, dtype=torch.uint8, device="cuda")
    with pytest.raises(p.AtrexError):
        agg.finalize(PEAK_BW, PEAK_FLOPS, out=out[: 48 * cap])
    assert (out[48 * cap:] == 0xA5).all()
