"""Depths 0 and 1 from one-hot planes and pair margins against the oracle.

Depth 1 counts only the cells with every value >= 1 and completes the table
from depth 0's pair tables; an item of its pool is a whole edge or a chunk of
ranks.  Covered: every pair of arities 2..5 (the counting shapes, with two
strata per pass or one), samples around the 64-sample word and across 65,536
(two counts per reduction below it), both statistics and both degrees of
freedom, values that never occur, pair tables from the Gram and from the
planes, an arity above 5 (histograms), enough edges for whole-edge items, and
edges whose lowest accepting rank many warps lower and read at once.
"""
import numpy as np
import pytest

import bnsynth
import oracle
from _compare import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2212_04259_gb300 import build
    build.build()
    import paper_2212_04259_gb300 as f
    return f


def _linked(seed, arities, N, drop=False):
    """Variables that follow a common one loosely: every pair dependent, so
    that depth 1 tests every triple."""
    rng = np.random.default_rng(seed)
    z = rng.integers(0, 5, N)
    rows = [np.where(rng.random(N) < 0.25, z % r, rng.integers(0, r, N)) for r in arities]
    if drop:
        rows[0] = np.minimum(rows[0], arities[0] - 2) if arities[0] > 2 else rows[0] * 0
        rows[-1] = np.maximum(rows[-1], 1)
    return np.stack(rows).astype(np.uint8), np.array(arities, dtype=np.uint8)


def _check(F, data, ar, alpha, md, stat="g2", df="fixed", **opt):
    ref = oracle.pc_stable(data, ar, alpha, md, stat=stat, df_mode=df)
    h = F.fbn_create(data, ar, statistic=stat, df=df, **opt)
    adj = F.fbn_learn_skeleton(h, alpha, md)
    hard, _, _ = compare(adj, F.fbn_export_sepsets(h), ref)
    assert not hard, hard[:3]
    st = F.fbn_get_stats(h)
    if not ref.near:
        assert st["tests_oracle"] == ref.tests and st["removed"] == ref.removed
    return st


@pytest.mark.parametrize("N", [63, 64, 65, 129, 2000, 65535, 65536, 70001])
@pytest.mark.parametrize("depth0", ["gram", "hist"])
def test_every_shape(F, N, depth0):
    data, ar = _linked(N, [2, 3, 4, 5, 5, 4, 3, 2, 4, 5], N)
    st = _check(F, data, ar, 0.05, 1, depth0=depth0)
    if st["depths"] > 1 and st["edges"][1]:
        assert st["popc_work"][1] > 0 and st["smem_updates"][1] == 0


@pytest.mark.parametrize("stat,df", [("g2", "adjusted"), ("x2", "fixed"), ("x2", "adjusted")])
@pytest.mark.parametrize("depth0", ["gram", "hist"])
def test_variants_and_missing_values(F, stat, df, depth0):
    for N, ars in ((3001, [5, 3, 2, 4, 5, 2, 3]), (66001, [3, 5, 4, 2, 3])):
        data, ar = _linked(N, ars, N, drop=True)
        _check(F, data, ar, 0.05, 1, stat, df, depth0=depth0)
        data, ar = _linked(N, [2] + ars[1:], N, drop=True)   # a constant variable
        _check(F, data, ar, 0.05, 1, stat, df, depth0=depth0)


def test_arity_above_the_planes_uses_histograms(F):
    data, ar = _linked(5, [6, 3, 4, 5, 2, 6], 5001)
    assert _check(F, data, ar, 0.05, -1)["popc_work"][1] == 0


@pytest.mark.parametrize("opt", [dict(), dict(group_size=3), dict(count="hist")])
def test_many_edges(F, opt):
    # about 80,000 edges at depth 1: whole-edge items by default
    rng = np.random.default_rng(3)
    probs = []
    for p in range(8):
        N = 1500 + 17 * p
        base = rng.integers(0, 3, N)
        rows = [np.where(rng.random(N) < 0.4, base % r, rng.integers(0, r, N)) for r in [2 + k % 3 for k in range(150)]]
        probs.append((np.stack(rows).astype(np.uint8), np.array([2 + k % 3 for k in range(150)], dtype=np.uint8)))
    hs = [F.fbn_create(d, a, **opt) for d, a in probs]
    adjs = F.fbn_learn_skeleton_batch(hs, 1e-4, 1)
    st = F.fbn_get_stats(hs[0])
    assert st["edges"][1] > 60000 and st["tests"][1] >= st["tests_oracle"][1]
    for p in (0, 7):
        d, a = probs[p]
        hard, _, _ = compare(adjs[p], F.fbn_export_sepsets(hs[p]), oracle.pc_stable(d, a, 1e-4, 1))
        assert not hard, hard[:3]


# 1,965 edges, each conditioning set an item of its own, and two edges in three have a set that
# accepts: warps read an edge's rank, and skip their item, while others lower it.
@pytest.mark.parametrize("opt", [dict(), dict(loop="host"), dict(group_size=1)])
def test_ranks_lowered_while_read(F, opt):
    rng = np.random.default_rng(11)
    N = 700
    base = rng.integers(0, 3, N)
    ar = np.array([2 + k % 3 for k in range(64)], dtype=np.uint8)
    data = np.stack([np.where(rng.random(N) < 0.45, base % r, rng.integers(0, r, N)) for r in ar]).astype(np.uint8)
    ref = oracle.pc_stable(data, ar, 1e-3, 1)
    h = F.fbn_create(data, ar, **opt)
    for _ in range(50):
        adj = F.fbn_learn_skeleton(h, 1e-3, 1)
        hard, _, _ = compare(adj, F.fbn_export_sepsets(h), ref)
        assert not hard, hard[:3]
        st = F.fbn_get_stats(h)
        assert st["tests_oracle"] == ref.tests and st["removed"] == ref.removed
    assert st["edges"][1] > 1000 and st["removed"][1] > 0
