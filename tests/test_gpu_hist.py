"""The histogram pools and the n ln n decision against the oracle.

Tables in interleaved copies at every group size, from a copy per lane to
one; tables around a warp's, a CTA's and the big class's shared memory and in
global memory; sample counts around the 16-sample vectors and two vectors per
thread; the same skeletons without the n ln n table (Pearson's statistic,
observed-table df) and in the edge-level form.
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


def _data(N, arities, keep, seed):
    """Every variable follows a common one, so that the edges survive to the
    deeper depths."""
    rng = np.random.default_rng(seed)
    base = rng.integers(0, 64, N)
    return np.stack([np.where(rng.random(N) < keep, base % r, rng.integers(0, r, N)) for r in arities]
                    ).astype(np.uint8), np.array(arities, dtype=np.uint8)


def _check(F, data, ar, alpha, md, stat="g2", df="fixed", **opt):
    ref = oracle.pc_stable(data, ar, alpha, md, stat=stat, df_mode=df)
    h = F.fbn_create(data, ar, statistic=stat, df=df, **opt)
    adj = F.fbn_learn_skeleton(h, alpha, md)
    hard, _, _ = compare(adj, F.fbn_export_sepsets(h), ref)
    assert not hard, hard[:3]
    if not ref.near:
        assert F.fbn_get_stats(h)["tests_oracle"] == ref.tests


@pytest.mark.parametrize("gt", [0, 32, 64, 128, 256])
@pytest.mark.parametrize("N", [15, 17, 511, 513, 1025, 16400])
def test_groups_and_ragged_samples(F, gt, N):
    data, ar = _data(N, [2, 3, 6, 2, 4, 3], 0.4, N)
    _check(F, data, ar, 0.3, -1, group_threads=gt, count="hist")


@pytest.mark.parametrize("stat,df", [("g2", "fixed"), ("x2", "fixed"), ("g2", "adjusted")])
@pytest.mark.parametrize("arities", [[16] * 4, [9, 8, 7, 20, 12], [24, 25, 26, 2], [12, 12, 12, 12, 3],
                                     [40, 41, 39, 3]])
def test_table_sizes(F, arities, stat, df):
    # bounds r_i r_j max^d from a few hundred cells to 69,000 at depths 1 and 2
    data, ar = _data(3001, arities, 0.5, sum(arities))
    _check(F, data, ar, 0.2, 2, stat, df)


def test_plain_form_and_large_counts(F):
    data, ar = _data(70001, [2, 6, 3, 4], 0.2, 9)
    for form in ("pool", "plain"):
        _check(F, data, ar, 0.05, -1, form=form)
