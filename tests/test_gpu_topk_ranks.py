"""The best k of a phase against Python integers, at the numbers of candidates where the ranking changes its way and for weighted
times that its scale cannot tell apart."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def weighted_times(n, law, rng):
    if law == "alike":
        return [5_000_000_007] * n
    if law == "nothing or one":
        return [int(x) for x in rng.integers(0, 2, n)]
    if law == "close":                      # one step of the scale, and low words that wrap around
        return [(1 << 64) - n // 2 + int(x) for x in rng.permutation(n)]
    return [(1 << int(b)) | int(rng.integers(0, 1 << 30)) for b in rng.integers(0, 88, n)]      # all magnitudes


@pytest.mark.parametrize("law", ["alike", "nothing or one", "close", "all magnitudes"])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 512, 513, 1_025, 2_047])
@pytest.mark.parametrize("max_keys", [4_096, 60_000])
def test_ranks_match_python(n, law, max_keys):
    import torch
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(n)
    entries = np.zeros(n, dtype=p.ENTRY_DTYPE)
    keys = (rng.permutation(4 * n)[:n].astype(np.uint64) << np.uint64(20)) | (np.uint64(1) << np.uint64(48))
    wt = weighted_times(n, law, rng)
    entries["key"], entries["count"] = keys, 1
    entries["wt_lo"], entries["wt_hi"] = [x & 0xFFFFFFFFFFFFFFFF for x in wt], [x >> 64 for x in wt]
    agg = p.Aggregator(np.ones(1, dtype=np.uint32), 2, max_keys)
    agg.merge(torch.from_numpy(entries.view(np.int64).reshape(n, 6)).cuda())
    agg.finalize(8e12, [1e15] * 8)
    order = sorted(range(n), key=lambda i: (-wt[i], int(keys[i])))
    for k in (1, 100, 512, 1_024):
        got = agg.topk(1, k)
        assert got["key"].tolist() == [int(keys[i]) for i in order[:k]]
        assert [int(e["wt_lo"]) | int(e["wt_hi"]) << 64 for e in got] == [wt[i] for i in order[:k]]
