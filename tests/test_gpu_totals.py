"""The totals pass at every number of phases a handle can have (its CTAs change shape from seven on)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3_000, 150_001])
@pytest.mark.parametrize("phases", range(1, 9))
def test_totals_counts_and_first_digits_of_every_phase(phases, n):
    """Merged entries of all eight phases -- those a handle's records cannot have included -- with weighted times from
    zero to 2^87, one phase without any: exact totals, key counts, and the best 700 by the digits counted on the way."""
    import torch
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(phases * 1000 + n)
    e = np.zeros(n, dtype=p.ENTRY_DTYPE)
    phase = rng.integers(0, 8, n).astype(np.uint64)
    phase[phase == 2] = 3
    e["key"] = phase << np.uint64(48) | np.arange(n, dtype=np.uint64) * np.uint64(7)
    e["count"] = rng.integers(1, 1000, n)
    bits = rng.integers(0, 64, n).astype(np.uint64)
    e["wt_lo"] = rng.integers(0, 1 << 64, n, dtype=np.uint64) >> bits
    e["wt_hi"] = np.where(bits < 8, rng.integers(0, 1 << 23, n), 0)
    e["wt_lo"][::17] = 0
    agg = p.Aggregator(np.ones(1, dtype=np.uint32), phases, max(n, 64))
    agg.merge(torch.from_numpy(e.view(np.uint8).reshape(-1)).cuda())
    got = agg.finalize_numpy(8e12, [1e15] * 8)
    assert len(got) == n
    lo, hi = agg.totals_words()
    keys = agg.stats()["keys_per_phase"]
    for q in range(8):
        rows = got[got["key"] >> np.uint64(48) == q]
        total = sum(int(x) for x in rows["wt_lo"]) + (sum(int(x) for x in rows["wt_hi"]) << 64)
        assert int(lo[q]) | int(hi[q]) << 64 == total and keys[q] == len(rows), q
        if q < phases:
            rows = rows[np.lexsort((rows["key"], ~rows["wt_lo"], ~rows["wt_hi"]))]
            for k in (1, 700):
                assert agg.topk(q, k).tobytes() == rows[:k].tobytes(), (q, k)
