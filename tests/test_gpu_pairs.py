"""Pair tables and depth-0 decisions from the Gram over the values >= 1.

The cells of value 0 follow from the single counts.  Covered: arities up to
255 (a lane per pair up to 8, a warp up to 32, a CTA of 256 threads up to 64 and of 1,024
above, narrow and wide problems in a batch), values that never occur, variable counts around the 32 pairs of a warp and
the 128 rows of a tile, output into host and device buffers, depth-0 decisions
with both statistics and both degrees of freedom, and depth 1 reading the
tables.  Counts and graphs equal to the oracle's.
"""
import numpy as np
import pytest

import oracle
from _compare import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2212_04259_gb300 import build
    build.build()
    import paper_2212_04259_gb300 as f
    return f


def _data(n, N, hi, seed):
    rng = np.random.default_rng(seed)
    ar = rng.integers(2, hi + 1, n).astype(np.uint8)
    base = rng.integers(0, 4, N)
    rows = [np.where(rng.random(N) < 0.1, base % r, rng.integers(0, r, N)) for r in ar]
    rows[0] = rows[0] * 0                       # a constant variable: value 0 only
    rows[1] = np.full(N, ar[1] - 1)             # ... its top value only
    rows[2] = np.maximum(rows[2], 1)            # value 0 never occurs
    return np.stack(rows).astype(np.uint8), ar


@pytest.mark.parametrize("n,N,hi", [(3, 1, 2), (31, 130, 5), (33, 8193, 24), (65, 300, 4), (130, 1000, 2),
                                    (24, 40000, 3), (200, 20011, 4), (9, 700, 9), (12, 3000, 32), (7, 5000, 33), (6, 900, 65),
                                    (5, 2001, 255)])   # few tiles of many samples: units of 8 stages and up
def test_pair_tables(F, n, N, hi):
    import torch
    data, ar = _data(n, N, hi, n + N)
    h = F.fbn_create(data, ar)
    M = int(ar.astype(int).sum())
    host = F.fbn_pairwise_counts(h)
    dev = torch.full((M, M), -1, dtype=torch.int32, device="cuda")
    F.fbn_pairwise_counts(h, dev)
    onehot = np.concatenate([(data[v][None, :] == np.arange(r)[:, None]) for v, r in enumerate(ar)]).astype(np.int64)
    assert np.array_equal(host, onehot @ onehot.T) and np.array_equal(dev.cpu().numpy(), host)


@pytest.mark.parametrize("stat,df", [("g2", "fixed"), ("g2", "adjusted"), ("x2", "fixed"), ("x2", "adjusted")])
@pytest.mark.parametrize("n,N,hi", [(33, 2000, 12), (70, 900, 5), (40, 66001, 5), (10, 3000, 8), (10, 3000, 9), (14, 70001, 32),
                                    (9, 30000, 33), (5, 70001, 255)])
def test_depth0_decisions(F, n, N, hi, stat, df):
    data, ar = _data(n, N, hi, 7 * n + N)
    ref = oracle.pc_stable(data, ar, 0.05, 1 if n < 50 and N < 5000 else 0, stat=stat, df_mode=df)
    h = F.fbn_create(data, ar, statistic=stat, df=df, depth0="gram")
    adj = F.fbn_learn_skeleton(h, 0.05, 1 if n < 50 and N < 5000 else 0)
    hard, _, _ = compare(adj, F.fbn_export_sepsets(h), ref)
    assert not hard, hard[:3]
    st = F.fbn_get_stats(h)
    assert st["edges"][0] == n * (n - 1) // 2 == st["tests"][0] and (ref.near or st["removed"] == ref.removed)


@pytest.mark.parametrize("stat,df", [("g2", "fixed"), ("x2", "adjusted")])
def test_batch_of_narrow_and_wide(F, stat, df):
    probs = [_data(n, N, hi, 3 * n) for n, N, hi in ((12, 2000, 4), (9, 3000, 20), (8, 4000, 60), (10, 1500, 8))]
    hs = [F.fbn_create(d, a, statistic=stat, df=df, depth0="gram") for d, a in probs]
    adjs = F.fbn_learn_skeleton_batch(hs, 0.05, 1)
    refs = [oracle.pc_stable(d, a, 0.05, 1, stat=stat, df_mode=df) for d, a in probs]
    for h, adj, ref in zip(hs, adjs, refs):
        hard, _, _ = compare(adj, F.fbn_export_sepsets(h), ref)
        assert not hard, hard[:3]
    st = F.fbn_get_stats(hs[0])
    assert st["edges"][0] == st["tests"][0] == sum(r.tests[0] for r in refs)
