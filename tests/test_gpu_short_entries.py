"""Short spill entries (8 bytes) and the directory's words form against the oracle: bit for bit, at the edges of their fields."""
import numpy as np
import pytest

import oracle
from tests.helpers import sorted_by_key
from tracegen.layout import RECORD_DTYPE

pytestmark = pytest.mark.gpu
PEAK_BW, PEAK_FLOPS = 8e12, [1e15] * 8


def check(agg, o):
    assert sorted_by_key(agg.finalize_numpy(PEAK_BW, PEAK_FLOPS)).tobytes() == o.finalize(PEAK_BW, PEAK_FLOPS).tobytes()


def ingest(agg, recs, start=0):
    import torch
    agg.ingest(torch.from_numpy(recs[start:].view(np.uint8).reshape(-1)).cuda(), n=len(recs) - start)


@pytest.mark.parametrize("max_keys", [2_000_000, 4_000_000, 9_000_000, 18_000_000, 1 << 25])      # 256 ... 4 096 partitions
@pytest.mark.parametrize("n_apps,n_phases,n_ops", [(1, 1, 1), (4, 2, 64), (4096, 2, 65), (300, 3, 128), (4096, 4, 256), (17, 8, 256), (4097, 2, 64)])
def test_every_field_at_its_edges(max_keys, n_apps, n_phases, n_ops):
    """Durations on both sides of every power of two (the longer ones take a second entry, from 2^16 to 2^31 on), the first
    and last application, phase and operator, shapes at the ends of their range, and three records whose operator is
    larger than any that a sample is likely to see."""
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(max_keys + n_apps)
    n, pool = 400_003, 60_000
    recs = np.zeros(n, dtype=RECORD_DTYPE)
    shapes = rng.integers(0, 1 << 32, pool, dtype=np.uint64).astype(np.uint32)
    shapes[:4] = (0, 1, 0x80000000, 0xFFFFFFFF)
    pick = np.where(rng.random(n) < 0.3, rng.integers(0, 300, n), rng.integers(0, pool, n))
    recs["shape_id"], recs["op_id"] = shapes[pick], pick % n_ops
    recs["app_id"] = np.where(rng.random(n) < 0.2, n_apps - 1, rng.integers(0, n_apps + 1, n))      # one in n_apps + 1 does not exist
    recs["phase"] = rng.integers(0, n_phases, n)
    edge = (np.uint64(1) << rng.integers(0, 33, n, dtype=np.uint64)) - rng.integers(0, 2, n, dtype=np.uint64)
    recs["duration_ns"] = np.minimum(edge, 0xFFFFFFFF).astype(np.uint32)
    recs["op_id"][[777, 200_000, n - 1]] = (n_ops, 0x0FFF, 0xFFFF)
    weights = rng.integers(0, 1 << 20, n_apps).astype(np.uint32)
    weights[-1] = 0xFFFFFFFF
    agg = p.Aggregator(weights, n_phases, max_keys)
    o = oracle.Oracle(weights, n_phases)
    for part in np.array_split(recs, [280_000]):                   # the second call meets the first one's keys, drained once
        ingest(agg, part)
        o.ingest(part, threads=4)
        check(agg, o)
    st = agg.stats()
    assert st["n_dropped"] == 0 and st["n_spilled"] <= st["n_valid"] and st["n_valid"] + st["n_rejected"] == n


@pytest.mark.parametrize("n_keys", [1, 3, 40])
def test_crowded_partitions_and_full_buffers(n_keys):
    """A second call whose records all go to a few keys that the directory does not hold: the partition pass sums equal
    entries first, and the buffers of one or two entries a record run over into the exact slow path."""
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(n_keys)
    n = (1 << 22) + 4096
    recs = np.zeros(n + (1 << 20), dtype=RECORD_DTYPE)
    recs["app_id"] = rng.integers(0, 3, len(recs))
    recs["op_id"], recs["shape_id"] = rng.integers(0, 5, len(recs)), rng.integers(0, 8_000, len(recs))
    recs["duration_ns"] = rng.choice(np.array([7, 0x00FFFFFF, 0x0FFFFFFF, 0xFFFFFFFF], dtype=np.uint32), len(recs))
    late = recs[n:]
    late["op_id"], late["shape_id"] = 6, 100_000 + rng.integers(0, n_keys, len(late))
    weights = np.array([1, 0xFFFF, 77], dtype=np.uint32)
    agg = p.Aggregator(weights, 1, 60_000)
    o = oracle.Oracle(weights, 1)
    o.ingest(recs, threads=8)
    ingest(agg, recs[:n])
    ingest(agg, recs, n)
    check(agg, o)
    st = agg.stats()
    assert st["n_valid"] == len(recs) and (st["n_overflow"] > 0) == (n_keys < 40)


def test_operators_that_no_longer_fit():
    """Records whose operator the sampled ones did not announce go to the table one by one until there are many; the
    entries are long from then on, the directory's sums so far are kept."""
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(5)
    n, part = 3 << 20, 1 << 20
    recs = np.zeros(n, dtype=RECORD_DTYPE)
    recs["app_id"], recs["phase"] = rng.integers(0, 9, n), rng.integers(0, 2, n)
    recs["op_id"], recs["shape_id"] = rng.integers(0, 100, n), rng.integers(0, 1000, n)
    recs["duration_ns"] = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
    recs["op_id"][part:] += np.where(rng.random(n - part) < 0.5, 5000, 0).astype(np.uint16)
    weights = rng.integers(0, 1 << 16, 9).astype(np.uint32)
    agg = p.Aggregator(weights, 2, 3_000_000)
    o = oracle.Oracle(weights, 2)
    for at in range(0, n, part):
        ingest(agg, recs[at: at + part])
        o.ingest(recs[at: at + part], threads=4)
    drains, cap = agg.stats()["n_drains"], agg.stats()["spill_cap"]
    check(agg, o)
    assert drains >= 2 and agg.stats()["n_valid"] == n
    agg.reset()                                                   # short entries again
    ingest(agg, recs[:part])
    assert agg.stats()["spill_cap"] == cap // 2 * 3


@pytest.mark.parametrize("hot", [0.0, 0.9])
@pytest.mark.parametrize("long_share", [0.7, 0.8, 1.0])
def test_durations_that_mostly_take_two_entries(long_share, hot):
    """Around the share of long durations from which the entries beside a dominant key are long ones (64 applications:
    26 bits or fewer fit a short entry)."""
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(int(long_share * 10 + hot * 100))
    n = 1_000_003
    recs = np.zeros(n, dtype=RECORD_DTYPE)
    recs["app_id"], recs["op_id"] = rng.integers(0, 64, n), rng.integers(0, 64, n)
    recs["phase"], recs["shape_id"] = rng.integers(0, 2, n), rng.integers(0, 8_192, n)
    cold = rng.random(n) >= hot
    for field in ("op_id", "phase", "shape_id"):
        recs[field] *= cold
    recs["duration_ns"] = np.where(rng.random(n) < long_share, (1 << 28) - 1, 50_000)
    weights = np.full(64, (1 << 20) - 1, dtype=np.uint32)
    agg = p.Aggregator(weights, 2, 2_000_000)
    o = oracle.Oracle(weights, 2)
    for _ in range(2):
        ingest(agg, recs)
        o.ingest(recs, threads=4)
    check(agg, o)


@pytest.mark.parametrize("n_apps,n_ops,max_keys", [(3, 9, 60_000), (300, 64, 60_000), (1_025, 256, 300_000), (2_500, 200, 4_000_000)])
def test_what_lies_behind_the_last_entry_is_not_looked_at(n_apps, n_ops, max_keys, monkeypatch):
    """Ragged buffers in a workspace of all ones, and in one that held the long entries of an earlier trace: where the number of
    applications is no power of two, an application field read from there names none (the bounds-checked build
    would say so)."""
    import torch
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(n_apps)
    weights = rng.integers(0, 1 << 20, n_apps).astype(np.uint32)
    empty = torch.empty
    with monkeypatch.context() as m:
        m.setattr(torch, "empty", lambda *args, **kw: empty(*args, **kw).fill_(0xFF))
        agg = p.Aggregator(weights, 2, max_keys)
    # (fewer records of a small table go straight into it)
    least = (1 << 22) + 1 if max_keys < 1_000_000 else 270_000
    for wide in (0, 1, 0):                                         # operators of any size: long entries
        n = least + 2 * int(rng.integers(0, 5_000))
        recs = np.zeros(n, dtype=RECORD_DTYPE)
        recs["app_id"], recs["phase"] = rng.integers(0, n_apps, n), rng.integers(0, 2, n)
        recs["op_id"], recs["shape_id"] = rng.integers(0, n_ops, n) + 60_000 * wide, rng.integers(0, max_keys // (3 * n_ops), n)
        recs["duration_ns"] = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32)
        o = oracle.Oracle(weights, 2)
        o.ingest(recs, threads=8)
        agg.reset()
        ingest(agg, recs)
        check(agg, o)
        st = agg.stats()
        assert 0 < st["n_spilled"] and st["n_valid"] == n


@pytest.mark.parametrize("hot", [0.0, 0.4, 0.9])
@pytest.mark.parametrize("long_share,is_short", [(0.0, True), (0.1, True), (0.6, False), (1.0, False)])
def test_entries_are_long_where_many_durations_take_two(long_share, is_short, hot):
    """The form of the entries, as the capacity of a buffer tells it, whatever the share of the most frequent key."""
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(int(long_share * 10 + hot * 100))
    n = 1_400_003                                                  # (below 2^20 it does not matter)
    recs = np.zeros(n, dtype=RECORD_DTYPE)
    recs["app_id"], recs["op_id"] = rng.integers(0, 64, n), rng.integers(0, 64, n)
    recs["phase"], recs["shape_id"] = rng.integers(0, 2, n), rng.integers(0, 8_192, n)
    cold = rng.random(n) >= hot
    for field in ("op_id", "phase", "shape_id"):
        recs[field] *= cold
    recs["duration_ns"] = np.where(rng.random(n) < long_share, (1 << 28) - 1, 50_000)
    agg = p.Aggregator(np.full(64, 7, dtype=np.uint32), 2, 2_000_000)
    cap = agg.stats()["spill_cap"]
    ingest(agg, recs)
    st = agg.stats()
    assert st["spill_cap"] == (cap // 2 * 3 if is_short else cap) and st["n_spilled"] > 0


def test_a_directory_is_built_anew_where_operators_no_longer_fit():
    """500 keys hold most of the trace.  When half of its records turn to operators that do not fit, the directory is given up;
    the call after that finds one for the records as they are now, and a reset starts afresh."""
    import torch
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(11)
    part = (1 << 20) + 5
    recs = np.zeros(4 * part, dtype=RECORD_DTYPE)
    recs["app_id"], recs["phase"] = rng.integers(0, 9, len(recs)), rng.integers(0, 2, len(recs))
    recs["op_id"] = rng.integers(0, 5, len(recs))
    recs["shape_id"] = np.where(rng.random(len(recs)) < 0.9, rng.integers(0, 50, len(recs)), rng.integers(50, 100_000, len(recs)))
    recs["duration_ns"] = rng.integers(0, 1 << 20, len(recs))
    recs["op_id"][part:] += np.where(rng.random(len(recs) - part) < 0.5, 5_000, 0).astype(np.uint16)
    weights = rng.integers(0, 1 << 16, 9).astype(np.uint32)
    agg = p.Aggregator(weights, 2, 3_000_000)
    for _ in range(2):
        o = oracle.Oracle(weights, 2)
        held, spilled = [], [0]
        for at in range(0, len(recs), part):
            ingest(agg, recs[at: at + part])
            o.ingest(recs[at: at + part], threads=4)
            torch.cuda.synchronize()
            held.append(agg.hot_directory() >> np.uint64(32) & np.uint64(0xFFFF))
            st = agg.stats()
            spilled.append(st["n_spilled"])
            assert st["hot_slots"] == len(held[-1]) and st["max_spill_fill"] <= st["spill_cap"]
        check(agg, o)
        assert len(held[0]) >= 490 and held[0].max() < 5
        assert len(held[1]) == 0
        assert all((h < 5).sum() >= 490 and (h >= 5_000).sum() >= 490 for h in held[2:])
        assert spilled[4] - spilled[3] < 0.2 * part
        agg.reset()


def test_buffers_have_room_for_two_entries_a_record():
    """Equally frequent keys, the first call's durations short, all others long, in calls of unequal size that leave the buffers
    just below the line that short durations are drained at: the full launch that follows must find room."""
    import torch
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(5)
    n, n_keys = 1 << 25, 500_000                                   # (records of one launch of such a table)
    recs = np.zeros(n, dtype=RECORD_DTYPE)
    recs["app_id"], recs["shape_id"] = rng.integers(0, 64, n), rng.integers(0, n_keys, n)
    recs["op_id"] = recs["shape_id"] % 7
    recs["duration_ns"] = (1 << 28) - 1
    few = recs[: (1 << 22) + 64].copy()                          # (fewer go straight into the table)
    few["duration_ns"] = 50_000
    weights = np.arange(1, 65, dtype=np.uint32)
    agg = p.Aggregator(weights, 2, 1_000_000)
    o = oracle.Oracle(weights, 2)
    cap = agg.stats()["spill_cap"]
    ingest(agg, few)
    o.ingest(few, threads=8)
    on_gpu = torch.from_numpy(recs.view(np.uint8).reshape(-1)).cuda()
    for part in (n, n, n // 8, n):
        agg.ingest(on_gpu, n=part)
        o.ingest(recs[:part], threads=8)
    st = agg.stats()
    assert st["spill_cap"] == cap // 2 * 3 and st["n_spilled"] > 0.9 * st["n_valid"]
    assert st["n_overflow"] == 0
    check(agg, o)


def test_fill_and_capacity_are_told_in_the_same_entries():
    """Buffers that ran over with short entries, whose capacity counts long ones after operators that do not fit."""
    import paper_2607_14541_b200 as p
    rng = np.random.default_rng(6)
    first, crowd, wide = (1 << 22) + 1, 1 << 20, 600_000
    recs = np.zeros(first + crowd + wide, dtype=RECORD_DTYPE)
    recs["op_id"], recs["shape_id"] = rng.integers(0, 5, len(recs)), rng.integers(0, 50_000, len(recs))
    recs["duration_ns"] = 1_000
    recs["op_id"][first: first + crowd], recs["shape_id"][first: first + crowd] = 6, 77_777
    recs["op_id"][first + crowd:] += 5_000
    weights = np.array([3], dtype=np.uint32)
    agg = p.Aggregator(weights, 1, 300_000)
    o = oracle.Oracle(weights, 1)
    o.ingest(recs, threads=8)
    cap = agg.stats()["spill_cap"]
    ingest(agg, recs[:first])
    ingest(agg, recs[first: first + crowd])
    st = agg.stats()
    assert st["spill_cap"] == st["max_spill_fill"] == cap // 2 * 3 and st["n_overflow"] > 0
    ingest(agg, recs, first + crowd)
    st = agg.stats()
    assert st["spill_cap"] == st["max_spill_fill"] == cap
    check(agg, o)


def test_the_largest_table_filled():
    """As many keys as the largest table is provisioned for, those of an (operator, shape) in all eight phases, with the weights of
    4 096 applications beside a partition's slots in shared memory (the least slots a key can have): none is dropped."""
    import torch
    import paper_2607_14541_b200 as p
    n, phases = 1 << 25, 8
    key = torch.arange(n, device="cuda")
    pair = key // phases
    recs = torch.empty(n, 4, dtype=torch.int32, device="cuda")
    recs[:, 0] = key % 4096
    recs[:, 1] = pair % 200 | (key % phases) << 16
    recs[:, 2] = pair // 200 * 2654435761 % (1 << 31)
    recs[:, 3] = 1_000
    agg = p.Aggregator(np.full(4096, 5, dtype=np.uint32), phases, n)
    for half in (recs[: n // 3], recs[n // 3:], recs):              # new keys beside old ones, then all of them found again
        agg.ingest(half)
        agg.stats()
    st = agg.stats()
    assert st["n_keys"] == n and st["n_dropped"] == 0 and st["keys_per_phase"][:phases] == [n // phases] * phases
    assert st["table_slots"] < 1.31 * n
    assert st["totals"][:phases] == [2 * n // phases * 5 * 1_000] * phases
