"""Critical values: an edge is removed exactly when p > alpha.

Two variables, alpha a part in 10^9 below and above the pair's own p-value, so
the decision turns on the critical value of that (df, alpha) being right to
about 10 digits (p and the critical value are both good to 13): degrees of
freedom from 1 to 529, p from strong dependence (far upper tail) to none (lower
tail), every way depth 0 is counted.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth0", ["auto", "gram", "hist"])
@pytest.mark.parametrize("rx,ry", [(2, 2), (2, 3), (5, 5), (7, 12), (24, 24)])
def test_decision_turns_at_p(rx, ry, depth0):
    import paper_2212_04259_gb300 as F
    rng = np.random.default_rng(rx * 100 + ry)
    ar = np.array([rx, ry], np.uint8)
    seen = 0
    for N, dep in [(400, 0.0), (3000, 0.02), (3000, 0.3), (500, 0.9), (20000, 0.0)]:
        x = rng.integers(0, rx, N)
        y = np.where(rng.random(N) < dep, x % ry, rng.integers(0, ry, N))
        data = np.stack([x, y]).astype(np.uint8)
        p = oracle.ci_test(data, ar, 0, 1, [])[2]
        if not 1e-250 < p < 1 - 1e-4:
            continue
        seen += 1
        step = 1e-9 * min(p, 1 - p)
        for alpha, kept in [(p - step, 0), (p + step, 1)]:
            h = F.fbn_create(data, ar, depth0=depth0)
            assert F.fbn_learn_skeleton(h, alpha, 0)[0, 1] == kept, (N, dep, p)
    assert seen >= 2
