"""Timed cases of the library's public entry points: what its users run, over the sizes they run it at.

Five paths, each called through the package as a user's program calls it:

  trace    device-resident records -> reset, ingest (one or many calls), finalize, the entry list in
           key order, top-k of every phase: one build of the benchmark's weights
  host     the same from records in pinned host memory (``ingest_host``)
  refresh  stored entry lists folded into a handle (``merge``), finalize, every phase ranked with its
           cumulative share and coverage cut
  weights  operator weights per Eq. 2-3 with per-application denominators
  score    Eq. 4-6 for a batch of candidates

A case is a dict of sizes and options; ``prepare`` makes its inputs on the GPU from a seed, and the output
buffers and scratch that such a program keeps between passes (rows behind a list's end stay zero).
"""
from __future__ import annotations

import ctypes
import math
import types

import numpy as np
import torch

import paper_2607_14541_b200 as p

PEAK_BW = 8.0e12
PEAK_FLOPS = (1.0e15, 2.0e15, 4.0e15)
PIECE = 1 << 25          # records made at a time


def _trace(name, records, calls, apps, ops, shapes, phases, zipf=0.0, live=0, hot=0.0, topk=10, path="trace"):
    """``shapes`` per operator drawn Zipf(``zipf``) (0: uniformly); ``live`` > 0: the keys are a list of that many
    (operator, shape, phase) triples out of the whole domain, drawn Zipf(``zipf``); ``hot``: share of the records
    that one key holds."""
    case = {"path": path, "records": records, "calls": calls, "apps": apps, "ops": ops, "shapes": shapes,
            "phases": phases, "zipf": zipf, "live": live, "hot": hot, "topk": topk}
    return dict(case, name=name) if name else case


def listed():
    return [
        # a few seconds of one service's trace: the latency of a whole build decides
        _trace("window_4k", 4_001, 1, 8, 32, 64, 2),
        # the tiny benchmark configuration: 2^20 records, uniform over 4 096 keys
        _trace("tiny_1m", 1 << 20, 1, 8, 32, 64, 2),
        # a collector that hands over its buffer every 4 K records or so: many small calls, ragged and unaligned
        _trace("stream_1m", 1_000_003, 244, 64, 48, 500, 2, zipf=1.1),
        # a day of one cluster: 2^26 records, 1 024 applications, Zipf(1.2) shapes
        _trace("zipf_64m", 1 << 26, 1, 1024, 64, 4096, 2, zipf=1.2),
        # high cardinality: 2^28 records over 2^22 live keys of three phases, the best 512 per phase
        _trace("highcard_256m", 1 << 28, 1, 256, 256, 1 << 20, 3, zipf=0.8, live=1 << 22, topk=512),
        # the headline configuration: 2^30 records in eight calls, 16 M keys
        _trace("chunked_1b", 1 << 30, 8, 4096, 128, 65536, 2, zipf=1.1),
        # one decode kernel dominates: 90 % of the records on one key
        _trace("skew_512m", 1 << 29, 1, 64, 64, 16384, 2, hot=0.9),
        # records still in (pinned) host memory
        _trace("host_20m", 20_000_003, 1, 1024, 64, 4096, 2, zipf=1.2, path="host"),
        # four stored weight lists brought together and ranked for release
        {"name": "refresh_5m", "path": "refresh", "lists": 4, "entries": 1_300_001, "domain": 1 << 22, "phases": 2,
         "coverage_ppm": 900_000},
        # Eq. 2-3 as written over 4 096 applications
        {"name": "weights_256m", "path": "weights", "records": (1 << 28) + 1, "calls": 2, "apps": 4096, "ops": 128,
         "shapes": 64, "phases": 2},
        # scoring many candidates at the paper's release size (440 units, 30 operators)
        {"name": "score_release", "path": "score", "candidates": 65_536, "units": 440, "ops": 30},
        # a few candidates over a wide suite with large operator groups
        {"name": "score_wide", "path": "score", "candidates": 1_000, "units": 12_001, "ops": 7},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def draw(rng):
    path = rng.choice(["trace"] * 8 + ["host"] * 2 + ["refresh"] * 3 + ["weights"] * 3 + ["score"] * 4)
    if path in ("trace", "host"):
        records = _log_int(rng, 1_000, 30_000_000 if path == "host" else 1_000_000_000)
        calls = _log_int(rng, 1, min(256, max(1, records // 1000)))
        apps, ops, phases = _log_int(rng, 4, 4096), _log_int(rng, 8, 256), rng.choice([1, 2, 2, 2, 3, 4])
        law = rng.choice(["zipf", "zipf", "zipf", "uniform", "live", "hot"])
        most = min(1 << 24, max(4096, 4 * records))                # distinct keys a trace of this size is set up for
        live, zipf, hot = 0, 0.0, 0.0
        if law == "live":
            records = min(records, 1 << 29)
            live, zipf, shapes = _log_int(rng, 1024, min(1 << 22, most)), rng.uniform(0.5, 1.0), 1 << 20
        else:
            shapes = _log_int(rng, 16, max(17, min(1 << 17, most // (ops * phases))))
            if law == "zipf":
                zipf = rng.uniform(0.8, 1.4)
            if law == "hot":
                hot = rng.uniform(0.3, 0.95)
        return _trace("", records, calls, apps, ops, shapes, phases, round(zipf, 3), live, round(hot, 3),
                      rng.choice([1, 10, 10, 100, 512]), path)
    if path == "refresh":
        lists, entries = rng.randint(1, 8), _log_int(rng, 1_000, 2_000_000)
        domain = min(1 << 24, int(entries * rng.uniform(1.1, 4.0)))
        return {"path": path, "lists": lists, "entries": entries, "domain": domain, "phases": rng.choice([1, 2, 2, 3, 4]),
                "coverage_ppm": rng.choice([0, 500_000, 900_000, 990_000])}
    if path == "weights":
        records = _log_int(rng, 10_000, 1 << 28)
        return {"path": path, "records": records, "calls": _log_int(rng, 1, min(64, max(1, records // 5000))),
                "apps": _log_int(rng, 4, 8192), "ops": _log_int(rng, 4, 256), "shapes": 64,
                "phases": rng.choice([1, 2, 2, 3])}
    units = _log_int(rng, 30, 16_384)
    return {"path": path, "candidates": max(1, _log_int(rng, 1, 30_000_000) // units), "units": units,
            "ops": min(units, _log_int(rng, 4, 300))}


# ---------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 1)
    return g


def _zipf_cdf(n, s):
    c = np.cumsum(np.arange(1, n + 1, dtype=np.float64) ** -s)      # (on the host: a parallel scan of floats may vary)
    return torch.from_numpy(c / c[-1]).cuda()


def _phase_shares(phases):
    """A third of the records is prefill, the rest is spread over the other phases."""
    return [1.0] if phases == 1 else [0.3] + [0.7 / (phases - 1)] * (phases - 1)


def _live_triples(case, ranks):
    """rank -> (phase, operator, shape): an affine map over the domain, so that every rank is another key."""
    domain = case["phases"] * case["ops"] * case["shapes"]
    a = int(domain * 0.6180339887) | 1
    while math.gcd(a, domain) != 1:
        a += 2
    t = (ranks * a + 12_345) % domain
    per_phase = case["ops"] * case["shapes"]
    rem = t % per_phase
    return t // per_phase, rem // case["shapes"], rem % case["shapes"]


def _app_weights(apps, g):
    """Card-hour weights: Zipf(1.1) over the applications, in a random order."""
    rank = torch.randperm(apps, generator=g, device="cuda").double() + 1
    return torch.clamp(((1 << 20) - 1) * rank.pow(-1.1), min=1).floor().to(torch.int64).cpu().numpy().astype(np.uint32)


def _durations(n, g):
    """Device times of production kernels: log-normal around 50 us."""
    d = torch.randn(n, generator=g, device="cuda", dtype=torch.float32).mul_(1.5).add_(math.log(5e4)).exp_()
    return d.clamp_(1000, (1 << 28) - 256).to(torch.int32)


def _records(case, g):
    """int32 [records, 4]: application, operator | phase << 16, shape, duration."""
    n, ops, shapes = case["records"], case["ops"], case["shapes"]
    out = torch.empty(n, 4, dtype=torch.int32, device="cuda")
    ranks = case.get("live") or shapes
    zipf, hot = case.get("zipf", 0.0), case.get("hot", 0.0)
    cdf = _zipf_cdf(ranks, zipf) if zipf else None
    shift = torch.randint(0, shapes, (ops,), generator=g, device="cuda")       # which shapes are frequent differs by operator
    bounds = torch.tensor(np.cumsum(_phase_shares(case["phases"]))[:-1], dtype=torch.float32, device="cuda")
    for lo in range(0, n, PIECE):
        m = min(PIECE, n - lo)
        if cdf is not None:
            rank = torch.searchsorted(cdf, torch.rand(m, generator=g, device="cuda", dtype=torch.float64)).clamp_(max=ranks - 1)
        else:
            rank = torch.randint(0, ranks, (m,), generator=g, device="cuda")
        if case.get("live"):
            phase, op, shape = _live_triples(case, rank)
        else:
            op = torch.randint(0, ops, (m,), generator=g, device="cuda")
            phase = torch.bucketize(torch.rand(m, generator=g, device="cuda"), bounds)
            shape = (rank + shift[op]) % shapes
        if hot:
            cold = torch.rand(m, generator=g, device="cuda") >= hot
            phase = torch.where(cold, phase, case["phases"] - 1)
            op, shape = op * cold, shape * cold
        piece = out[lo: lo + m]
        piece[:, 0] = torch.randint(0, case["apps"], (m,), generator=g, device="cuda", dtype=torch.int32)
        piece[:, 1] = op | (phase << 16)
        piece[:, 2] = shape
        piece[:, 3] = _durations(m, g)
    return out


def _work_table(case, g):
    """One row per (operator, shape) in use: flops and bytes log-uniform in [1e6, 1e13], three dtypes."""
    ops, shapes = case["ops"], case["shapes"]
    if case.get("live"):
        _, op, shape = _live_triples(case, torch.arange(case["live"], device="cuda"))
        pair = torch.unique(op * shapes + shape)
    else:
        pair = torch.arange(ops * shapes, device="cuda")
    m = pair.numel()
    rows = torch.empty(m, 3, dtype=torch.int64, device="cuda")
    dtype = torch.randint(0, len(PEAK_FLOPS), (m,), generator=g, device="cuda")
    rows[:, 0] = (pair % shapes) | ((pair // shapes) << 32) | (dtype << 48)
    for col in (1, 2):
        rows[:, col] = torch.pow(10.0, 6 + 7 * torch.rand(m, generator=g, device="cuda", dtype=torch.float64)).to(torch.int64)
    return rows.cpu().numpy().reshape(-1).view(p.WORK_DTYPE)


def _provisioned_keys(case):
    return case["live"] or case["ops"] * case["shapes"] * case["phases"]


def _calls(records, calls):
    """The records split into ``calls`` consecutive slices."""
    n = records.shape[0]
    at = [n * c // calls for c in range(calls + 1)]
    return [records[a:b] for a, b in zip(at, at[1:]) if b > a]


def _entry_buffer(rows):
    return torch.zeros(rows * 48, dtype=torch.uint8, device="cuda")


def _release_scratch(entries):
    return torch.empty(p.atrex_release_scratch_bytes(entries), dtype=torch.uint8, device="cuda")


def _prepare_trace(case, g):
    weights, work, records = _app_weights(case["apps"], g), _work_table(case, g), _records(case, g)
    keys = _provisioned_keys(case)
    agg = p.Aggregator(weights, case["phases"], keys, max_work_rows=len(work))
    agg.set_work_table(work)
    if case["path"] == "host":
        pinned = torch.empty(records.shape, dtype=torch.int32, pin_memory=True)
        pinned.copy_(records)
        records = pinned
    return types.SimpleNamespace(case=case, agg=agg, parts=_calls(records, case["calls"]), out=_entry_buffer(keys),
                                 by_key=_entry_buffer(keys), scratch=_release_scratch(keys))


def _prepare_refresh(case, g):
    lists, m, domain, phases = case["lists"], case["entries"], case["domain"], case["phases"]
    parts = []
    for _ in range(lists):
        t = torch.randperm(domain, generator=g, device="cuda")[:m]
        e = torch.zeros(t.numel(), 6, dtype=torch.int64, device="cuda")
        pair = t // phases
        e[:, 0] = (pair // 64) | ((pair % 64) << 32) | ((t % phases) << 48)
        e[:, 1] = torch.randint(1, 100_000, (t.numel(),), generator=g, device="cuda")
        mean = torch.randn(t.numel(), generator=g, device="cuda", dtype=torch.float64).mul_(2.5).add_(math.log(5e9)).exp_()
        e[:, 2] = (e[:, 1] * mean).clamp_(max=2.0 ** 60).to(torch.int64)
        parts.append(e)
    pairs = -(-domain // phases)
    t = torch.arange(pairs, device="cuda")
    rows = torch.empty(pairs, 3, dtype=torch.int64, device="cuda")
    rows[:, 0] = (t // 64) | ((t % 64) << 32)
    for col in (1, 2):
        rows[:, col] = torch.pow(10.0, 6 + 7 * torch.rand(pairs, generator=g, device="cuda", dtype=torch.float64)).to(torch.int64)
    agg = p.Aggregator(np.ones(1, dtype=np.uint32), phases, domain, max_work_rows=pairs)
    agg.set_work_table(rows.cpu().numpy().reshape(-1).view(p.WORK_DTYPE))
    # (a phase's keys are every phases-th of the domain: none has more than `pairs`)
    return types.SimpleNamespace(case=case, agg=agg, parts=parts, out=_entry_buffer(domain), scratch=_release_scratch(domain),
                                 ranked=[_entry_buffer(pairs) for _ in range(phases)],
                                 cum=[torch.zeros(pairs, dtype=torch.float64, device="cuda") for _ in range(phases)])


def _prepare_weights(case, g):
    records = _records(case, g)
    handle = p.OperatorWeights(_app_weights(case["apps"], g), case["ops"], case["phases"])
    retained = (torch.rand(case["ops"], generator=g, device="cuda") < 0.9).to(torch.uint8).cpu().numpy()
    return types.SimpleNamespace(case=case, handle=handle, parts=_calls(records, case["calls"]), retained=retained)


def _prepare_score(case, g):
    b, n, ops = case["candidates"], case["units"], case["ops"]

    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)

    roofline = torch.pow(10.0, -7 + 5 * rand(n))
    unit_op = torch.randint(0, ops, (n,), generator=g, device="cuda", dtype=torch.int32)
    t_cand = roofline / (0.02 + 0.95 * rand(b, n))                       # attained shares of the roofline
    odd = torch.randint(0, 100_000, (b, n), generator=g, device="cuda")  # now and then a faulty measurement
    t_cand = torch.where(odd == 0, roofline * 0.5, torch.where(odd == 1, 0.0, t_cand))
    correct = (rand(b, n) < 0.85).to(torch.uint8)
    w = rand(ops)
    return types.SimpleNamespace(case=case, args=(roofline, unit_op, t_cand, correct, w / w.sum()))


def prepare(case, seed):
    g = _generator(seed)
    make = {"trace": _prepare_trace, "host": _prepare_trace, "refresh": _prepare_refresh, "weights": _prepare_weights,
            "score": _prepare_score}
    return make[case["path"]](case, g)


# ---------------------------------------------------------------- one pass

def _rows(entries):
    return entries.view(torch.int64).view(-1, 6)


def _ok(status, where):
    if status != p.ATREX_OK:
        raise p.AtrexError(status, where)


def _build(state):
    """One build of the weights: the entries in key order and every phase's top-k."""
    case, agg = state.case, state.agg
    for part in state.parts:
        if case["path"] == "host":
            agg.ingest_host(part)
        else:
            agg.ingest(part)
    entries, n = agg.finalize(PEAK_BW, PEAK_FLOPS, out=state.out)
    _ok(p.atrex_entries_sort_by_key(entries.data_ptr(), n, state.by_key.data_ptr(), state.scratch.data_ptr(),
                                    state.scratch.numel(), torch.cuda.current_stream().cuda_stream),
        "atrex_entries_sort_by_key")
    top = [agg.topk(phase, case["topk"]).view(np.int64) for phase in range(case["phases"])]
    return {"n": n, "entries": _rows(state.by_key), "top": top}


def _refresh(state):
    """Stored lists folded together, every phase ranked for release."""
    case, agg = state.case, state.agg
    for part in state.parts:
        agg.merge(part)
    entries, n = agg.finalize(PEAK_BW, PEAK_FLOPS, out=state.out)
    result = []
    for phase in range(case["phases"]):
        cut, ranked, cum = p.atrex_rank_result_t(), state.ranked[phase], state.cum[phase]
        _ok(p.atrex_entries_rank(entries.data_ptr(), n, phase, case["coverage_ppm"], ranked.data_ptr(), cum.data_ptr(),
                                 cum.numel(), ctypes.byref(cut), state.scratch.data_ptr(), state.scratch.numel(),
                                 torch.cuda.current_stream().cuda_stream), "atrex_entries_rank")
        result.append([_rows(ranked), cum, cut.n_phase, cut.n_keep])
    return result


def run(state):
    path = state.case["path"]
    if path == "score":
        return p.score_aggregate(*state.args)
    if path == "weights":
        state.handle.reset()
        for part in state.parts:
            state.handle.ingest(part)
        return state.handle.finalize(retained=state.retained)
    state.agg.reset()
    return _refresh(state) if path == "refresh" else _build(state)


# ---------------------------------------------------------------- what a pass cannot do without

def _expected_keys(case):
    n = case["records"]
    if case["live"]:
        share = np.arange(1, case["live"] + 1, dtype=np.float64) ** -case["zipf"]
        return float(np.sum(-np.expm1(-n * share / share.sum())))
    share = np.arange(1, case["shapes"] + 1, dtype=np.float64) ** -case["zipf"]
    share /= share.sum()
    return float(sum(case["ops"] * np.sum(-np.expm1(-n * (1 - case["hot"]) * q / case["ops"] * share))
                     for q in _phase_shares(case["phases"])))


def work(case):
    """Every record (entry, time) read once, every result written once; a key's work-table row read once."""
    if case["path"] == "score":
        b, n, ops = case["candidates"], case["units"], case["ops"]
        return {"bytes": 9.0 * b * n + 12.0 * n + 8.0 * ops + 8.0 * b * (ops + 2), "flops": float(b * n)}
    if case["path"] == "weights":
        return {"bytes": 16.0 * case["records"] + 16.0 * case["ops"], "flops": float(case["records"])}
    if case["path"] == "refresh":
        lists, m, domain = case["lists"], min(case["entries"], case["domain"]), case["domain"]
        keys = domain * (1.0 - (1.0 - m / domain) ** lists)
        return {"bytes": 48.0 * lists * m + (24.0 + 56.0) * keys, "flops": 2.0 * lists * m + 4.0 * keys}
    keys = _expected_keys(case)
    return {"bytes": 16.0 * case["records"] + (24.0 + 48.0) * keys + 48.0 * case["topk"] * case["phases"],
            "flops": 2.0 * case["records"] + 4.0 * keys}


def tolerance(case):
    """Sums are integers and every floating-point step is one rounding in a fixed order: one bit pattern."""
    return "exact"
