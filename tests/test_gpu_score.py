"""Parity of the score-aggregation kernel (Eq. 4-6) with the oracle, bit for bit."""
import numpy as np
import pytest

import oracle
from tests.helpers import load_golden

pytestmark = pytest.mark.gpu


def run_gpu(roof, unit_op, t, ok, w):
    import torch
    import paper_2607_14541_b200 as p
    d = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a, dtype=dt)).cuda()
    s_agg, s_op, err = p.score_aggregate(d(roof, np.float64), d(unit_op, np.int32), d(t, np.float64),
                                         d(ok, np.uint8), d(w, np.float64))
    torch.cuda.synchronize()
    return s_agg.cpu().numpy(), s_op.cpu().numpy(), err.cpu().numpy().astype(np.uint64)


def test_score_worked_example_on_gpu(golden_dir):
    g = load_golden(golden_dir, "score_example.json")
    u = g["units"]
    agg, s_op, err = run_gpu([x["roofline_s"] for x in u], [x["op"] for x in u], [[x["t_cand"] for x in u]],
                             [[x["correct"] for x in u]], g["w"])
    assert list(s_op[0]) == g["S_op"] and float(agg[0]) == g["S_agg"] and int(err[0]) == g["errors"]


@pytest.mark.parametrize("n_ops,n_units,batch,seed", [(30, 440, 64, 0), (1, 1, 3, 1), (257, 5000, 17, 2), (4, 16384, 2, 3)])
def test_score_parity_random_batches(n_ops, n_units, batch, seed):
    rng = np.random.default_rng(seed)
    unit_op = rng.integers(0, n_ops, n_units).astype(np.uint32)            # unsorted on purpose
    if n_units > 10:
        unit_op[:3] = n_ops + 5                                           # out-of-range operators are ignored
    roof = np.exp(rng.uniform(np.log(1e-6), np.log(1e-1), n_units))
    w = rng.dirichlet(np.ones(n_ops))
    ratio = rng.uniform(0.01, 1.1, (batch, n_units))
    ratio[:, ::7] = 0.5                                                   # plenty of exact ties
    t = roof[None, :] / ratio
    ok = rng.random((batch, n_units)) < 0.6
    ok[0] = False                                                         # a candidate with nothing correct
    if n_units > 10:
        t[1, 4], t[1, 5], t[1, 6] = np.inf, -1.0, np.nan
        ok[1, 4:7] = True
    exp = oracle.score_candidates(roof, unit_op, t, ok, w)
    got = run_gpu(roof, unit_op, t, ok, w)
    assert got[0].tobytes() == exp[0].tobytes()
    assert got[1].tobytes() == exp[1].tobytes()
    assert np.array_equal(got[2], exp[2])
    assert float(got[0][0]) == 0.0


def test_score_limits():
    import torch
    import paper_2607_14541_b200 as p
    z = torch.zeros(8, dtype=torch.float64, device="cuda")
    assert p.atrex_score_aggregate(z.data_ptr(), z.data_ptr(), p.lib.atrex_score_aggregate.argtypes and 16385, z.data_ptr(),
                                   z.data_ptr(), 1, z.data_ptr(), 1, z.data_ptr(), None, None, None) == p.ATREX_ERR_TOO_LARGE
    assert p.atrex_score_aggregate(None, z.data_ptr(), 4, z.data_ptr(), z.data_ptr(), 1, z.data_ptr(), 1, z.data_ptr(),
                                   None, None, None) == p.ATREX_ERR_INVALID
    assert p.atrex_score_aggregate(None, None, 4, None, None, 0, None, 1, None, None, None, None) == p.ATREX_OK


# group sizes at the edges of the lane-sorted columns, the register searches and the shared-memory search
EDGE_GROUPS = {"lanes": [1, 2, 7, 8, 9, 15, 16, 17, 20, 24, 25, 28, 31, 32, 0, 5], "mixed": [32, 33, 3, 64, 65, 1, 128, 129, 0, 40],
               "wide": [255, 256, 257, 600, 31, 33], "many": [3, 0, 9, 1] * 40,
               "pairs": [33, 63, 64, 65, 40, 31, 1, 0, 2, 47, 48, 49, 56, 24, 25, 35, 60, 3, 32, 16, 130, 17]}


@pytest.mark.parametrize("batch", [3, 700, 2500])  # one candidate per CTA (small CTAs at 700 and up to 1 024 units), one per warp
@pytest.mark.parametrize("groups", sorted(EDGE_GROUPS))
def test_score_parity_at_group_size_edges(groups, batch):
    sizes = EDGE_GROUPS[groups]
    n_ops, n_units = len(sizes), sum(sizes)
    rng = np.random.default_rng(n_units + batch)
    unit_op = rng.permutation(np.repeat(np.arange(n_ops), sizes)).astype(np.uint32)
    roof = np.exp(rng.uniform(np.log(1e-6), np.log(1e-1), n_units))
    t = roof[None, :] / rng.uniform(0.01, 1.02, (batch, n_units))
    t[0::5] = roof / np.round(rng.uniform(0.1, 1.0, n_units), 1)          # ties
    t[1::5] = roof / 0.5 * (1 + rng.integers(0, 4, (len(t[1::5]), n_units)) * 2.0 ** -50)   # scores a few units in the last place apart
    t[2::5, : n_units // 2] *= 2.0 ** -100                                # far outside the usual range
    ok = rng.random((batch, n_units)) < 0.8
    t[3::5, ::9] = 0.0
    w = rng.dirichlet(np.ones(n_ops))
    exp = oracle.score_candidates(roof, unit_op, t, ok, w)
    got = run_gpu(roof, unit_op, t, ok, w)
    assert got[0].tobytes() == exp[0].tobytes()
    assert got[1].tobytes() == exp[1].tobytes()
    assert np.array_equal(got[2], exp[2])


@pytest.mark.parametrize("batch", [592, 593, 740, 741, 1_184, 1_185])
@pytest.mark.parametrize("n_units,n_ops", [(700, 28), (800, 22), (801, 27), (1_400, 56), (1_401, 40), (500, 10), (501, 16)])
def test_score_parity_where_the_kernels_change(n_units, n_ops, batch):
    """Candidates on both sides of what the SMs hold at once (CTAs of 256, 192 and 128 threads, one candidate per warp)."""
    rng = np.random.default_rng(n_units + batch)
    unit_op = rng.integers(0, n_ops + 1, n_units).astype(np.uint32)       # one operator in n_ops + 1 is out of range
    roof = np.exp(rng.uniform(np.log(1e-6), np.log(1e-1), n_units))
    t = roof[None, :] / rng.uniform(0.01, 1.02, (batch, n_units))
    t[0::5] = roof / np.round(rng.uniform(0.1, 1.0, n_units), 1)          # ties
    ok = rng.random((batch, n_units)) < 0.8
    w = rng.dirichlet(np.ones(n_ops))
    exp = oracle.score_candidates(roof, unit_op, t, ok, w)
    got = run_gpu(roof, unit_op, t, ok, w)
    assert got[0].tobytes() == exp[0].tobytes()
    assert got[1].tobytes() == exp[1].tobytes()
    assert np.array_equal(got[2], exp[2])


# operators counted by range: sizes around every line of its dispatch, groups that end in the first, the last and a crowded range
@pytest.mark.parametrize("n_units,n_ops,batch", [
    (64, 1, 3), (127, 2, 150), (128, 2, 150), (1000, 15, 149), (1001, 15, 149), (1000, 3, 600), (2001, 2, 300), (3000, 40, 20), (3001, 40, 20),
    (4001, 5, 460), (9001, 101, 150), (14_001, 7, 149), (16_320, 255, 2), (16_384, 256, 2), (16_384, 1, 150)])
@pytest.mark.parametrize("law", ["even", "uneven", "two values", "far apart", "close"])
def test_score_parity_by_counting(n_units, n_ops, batch, law):
    rng = np.random.default_rng(n_units + n_ops + len(law))
    unit_op = rng.integers(0, n_ops + 1, n_units).astype(np.uint32)       # one operator in n_ops + 1 is out of range
    if law == "uneven":
        unit_op[: n_units // 2] = n_ops - 1
    roof = np.exp(rng.uniform(np.log(1e-6), np.log(1e-1), n_units))
    batch = min(batch, 3_000_000 // n_units)
    score = rng.uniform(0.01, 1.02, (batch, n_units))
    if law == "two values":                                               # the middles lie in different ranges, or among ties
        score = np.where(rng.random((batch, n_units)) < 0.5, 0.01, 0.9)
    if law == "far apart":                                                # mostly outside the first cut's range
        score = np.exp2(rng.uniform(-50, 40, (batch, n_units)))
    if law == "close":
        score = 0.3 * (1 + rng.integers(0, 1 << 12, (batch, n_units)) * 2.0 ** -34)
    t = roof[None, :] / score
    if law == "far apart":
        t[:, ::501] *= 2.0 ** -300                                        # outside binary32
    t[0::7, ::9] = 0.0
    ok = rng.random((batch, n_units)) < 0.8
    ok[-1] = unit_op[None, :] == 0                                        # an operator or none with anything correct
    w = rng.dirichlet(np.ones(n_ops))
    exp = oracle.score_candidates(roof, unit_op, t, ok, w)
    got = run_gpu(roof, unit_op, t, ok, w)
    assert got[0].tobytes() == exp[0].tobytes()
    assert got[1].tobytes() == exp[1].tobytes()
    assert np.array_equal(got[2], exp[2])


@pytest.mark.parametrize("n_units,n_ops,batch", [(64, 1, 2_000), (700, 10, 2_000), (1_001, 15, 1_500), (4_001, 31, 700), (16_320, 255, 3), (16_384, 1, 3)])
def test_score_parity_where_operators_are_searched(n_units, n_ops, batch):
    """Operators whose keys do not tell the middle beside others of the same candidate, and candidates without any behind them: per operator
    and candidate, scores spread out, all alike, alike in their leading bits, of two values, or with one outside binary32."""
    rng = np.random.default_rng(n_units + n_ops)
    unit_op = rng.integers(0, n_ops, n_units).astype(np.uint32)
    roof = np.exp(rng.uniform(np.log(1e-6), np.log(1e-1), n_units))
    law = rng.integers(0, 5, (batch, n_ops))
    law[::3] = 0
    law = law[:, unit_op]
    score = rng.uniform(0.01, 1.02, (batch, n_units))
    score = np.where(law == 1, 0.25, score)
    score = np.where(law == 2, 0.3 * (1 + np.floor(score * 4096) * 2.0 ** -34), score)
    score = np.where(law == 3, np.where(score < 0.5, 0.01, 0.9), score)
    t = roof[None, :] / score
    t[law == 1] = np.broadcast_to(4.0 * roof, t.shape)[law == 1]         # (exactly one score)
    t[:, ::61] *= np.where(law[:, ::61] == 4, 2.0 ** -300, 1.0)
    ok = rng.random((batch, n_units)) < 0.8
    w = rng.dirichlet(np.ones(n_ops))
    exp = oracle.score_candidates(roof, unit_op, t, ok, w)
    got = run_gpu(roof, unit_op, t, ok, w)
    assert got[0].tobytes() == exp[0].tobytes()
    assert got[1].tobytes() == exp[1].tobytes()
    assert np.array_equal(got[2], exp[2])


@pytest.mark.parametrize("batch", [2_367, 2_368])
@pytest.mark.parametrize("n_units,n_ops", [(64, 1), (500, 1), (500, 7), (501, 7)])
def test_score_parity_between_counting_and_warps(n_units, n_ops, batch):
    """Large groups of few units: a CTA per candidate that counts them, or from 16 candidates per SM on a warp."""
    rng = np.random.default_rng(n_units + batch)
    unit_op = rng.integers(0, n_ops, n_units).astype(np.uint32)
    roof = np.exp(rng.uniform(np.log(1e-6), np.log(1e-1), n_units))
    t = roof[None, :] / rng.uniform(0.01, 1.02, (batch, n_units))
    t[0::5] = roof / np.round(rng.uniform(0.1, 1.0, n_units), 1)          # ties
    t[1::7] = roof / (0.3 * (1 + rng.integers(0, 1 << 12, n_units) * 2.0 ** -34))
    ok = rng.random((batch, n_units)) < 0.8
    w = rng.dirichlet(np.ones(n_ops))
    exp = oracle.score_candidates(roof, unit_op, t, ok, w)
    got = run_gpu(roof, unit_op, t, ok, w)
    assert got[0].tobytes() == exp[0].tobytes()
    assert got[1].tobytes() == exp[1].tobytes()
    assert np.array_equal(got[2], exp[2])
