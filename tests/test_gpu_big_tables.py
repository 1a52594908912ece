"""Big tables (above the small class's share of shared memory) against the oracle.

Covered: both kernels of the class (many tests and few, tables that fit the
256-thread kernel's shared memory, ones that only fit the 1,024-thread one's, and
ones that go to global memory), with and without marginals beside the table.
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


def _linked(seed, n, r, N, strength=0.3):
    rng = np.random.default_rng(seed)
    base = rng.integers(0, r, N)
    data = np.stack([np.where(rng.random(N) < strength, base, rng.integers(0, r, N)) for _ in range(n)]).astype(np.uint8)
    return data, np.full(n, r, np.uint8)


# cells at the deepest depth: 7,776; 20,736; 24,389 and 27,000 (the 256-thread kernel takes up to 25,600 ints); 64,000
@pytest.mark.parametrize("n,r,md", [(9, 6, 3), (8, 12, 2), (10, 29, 1), (10, 30, 1), (5, 30, 1), (9, 40, 1)])
@pytest.mark.parametrize("stat,df", [("g2", "fixed"), ("x2", "fixed"), ("g2", "adjusted"), ("x2", "adjusted")])
@pytest.mark.parametrize("loop", ["host", "device"])
def test_big_tables(F, n, r, md, stat, df, loop):
    data, ar = _linked(r, n, r, 20011 if r == 6 else 3001, 0.6 if r == 6 else 0.3)
    ref = oracle.pc_stable(data, ar, 0.05, md, stat=stat, df_mode=df)
    h = F.fbn_create(data, ar, statistic=stat, df=df, loop=loop)
    adj = F.fbn_learn_skeleton(h, 0.05, md)
    hard, _, _ = compare(adj, F.fbn_export_sepsets(h), ref)
    assert not hard, hard[:3]
    st = F.fbn_get_stats(h)
    assert all(0 < t <= m for t, m in zip(st["test_ms"], st["ms"])), st
    if not ref.near:
        assert st["tests_oracle"] == ref.tests and st["removed"] == ref.removed
