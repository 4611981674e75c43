"""Top-k where the one-CTA ranking does not do: k above 1 024, or thousands of keys level with the k-th."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
PEAK_BW, PEAK_FLOPS = 8e12, [1e15] * 8
PHASES = 5


def merged(law, n=200_000, seed=3):
    """A handle into which n entries are merged, a fiftieth of them of phase 4, and its entries by phase in ranking order."""
    import torch
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(seed)
    e = np.zeros(n, dtype=p.ENTRY_DTYPE)
    phase = np.where(np.arange(n) % 50 == 0, 4, np.arange(n) % 4).astype(np.uint64)
    e["key"] = phase << np.uint64(48) | (rng.permutation(n).astype(np.uint64) % np.uint64(997)) << np.uint64(32) | np.arange(n, dtype=np.uint64)
    e["count"] = 1
    if law == "spread":
        e["wt_lo"] = np.exp(rng.normal(22, 2.5, n)).astype(np.uint64)
    elif law == "flat":
        e["wt_lo"] = (1 << 40) + rng.integers(0, 1 << 20, n).astype(np.uint64)
    elif law == "equal":
        e["wt_lo"] = 12_345_678
    elif law == "small":
        e["wt_lo"] = rng.integers(0, 70, n)
    elif law == "wide":
        e["wt_lo"], e["wt_hi"] = rng.integers(0, 1 << 63, n), rng.integers(0, 1 << 4, n)
    agg = p.Aggregator(np.ones(1, dtype=np.uint32), PHASES, n)
    agg.merge(torch.from_numpy(e.view(np.uint8).reshape(-1)).cuda())
    got = agg.finalize_numpy(PEAK_BW, PEAK_FLOPS)
    by_phase = []
    for q in range(PHASES):
        rows = got[got["key"] >> np.uint64(48) == q]
        by_phase.append(rows[np.lexsort((rows["key"], ~rows["wt_lo"], ~rows["wt_hi"]))])
    return agg, by_phase


@pytest.mark.parametrize("law", ["spread", "flat", "equal", "small", "wide"])
def test_every_phase_is_ranked_exactly(law):
    """Weights over orders of magnitude, within a millionth of each other, all the same, zero among few values and beyond
    64 bits; k on both sides of the one-CTA ranking, of the sorter's powers of two, of a phase's keys and at the limit."""
    agg, by_phase = merged(law)
    assert [len(r) for r in by_phase][3:] == [50_000, 4_000]
    for k in (1, 1024, 1025, 2047, 2048, 4000, 4097, 49_999, 65_536):
        for q in range(PHASES):
            assert agg.topk(q, k).tobytes() == by_phase[q][:k].tobytes(), (k, q)


def test_one_selection_serves_every_phase():
    """The first request of a k selects for all phases -- in no more passes over the table than for one -- and the
    others only fetch their rows; another k reads the table again, but not for the first digit's counts."""
    agg, by_phase = merged("spread")
    for k in (1500, 3000):
        before = agg.launch_count()
        agg.topk(0, k)
        first = agg.launch_count() - before
        assert first <= 6                                    # digit, count, digit, collect, sort, rows
        for q in range(1, PHASES):
            before = agg.launch_count()
            agg.topk(q, k)
            assert agg.launch_count() - before == 1, q
