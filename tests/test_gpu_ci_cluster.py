"""Explicit tests on a thread-block cluster against the oracle.

A test runs on 1 to 16 CTAs by its samples and cells; each CTA counts a share
of the samples and reduces a share of the strata.  Covered: sample counts at
the edges of the cluster sizes and of the 16-sample vectors, fewer strata than
CTAs, tables in shared and in global memory, many cells on few samples (shares
without a sample), and the p-value on both sides of the mean for even and odd
degrees of freedom.  Counts bit-exact, G^2 within 1e-6 relative and p within
1e-9 absolute of the oracle.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2212_04259_gb300 import build
    build.build()
    import paper_2212_04259_gb300 as f
    return f


def _data(N, arities, dep):
    rng = np.random.default_rng(N + 7 * len(arities))
    rows = [rng.integers(0, r, N) for r in arities]
    if dep:   # X copied into Y now and then: the statistic above its mean
        rows[1] = np.where(rng.random(N) < dep, rows[0] % arities[1], rows[1])
    return np.stack(rows).astype(np.uint8), np.array(arities, dtype=np.uint8)


@pytest.mark.parametrize("arities,S", [([2, 2], []), ([2, 3, 2], [2]), ([5, 4, 3, 7], [3, 2]), ([4, 3, 5, 5, 5], [2, 4, 3]),
                                       ([16, 15, 17, 9], [2, 3]), ([9, 8, 30, 31], [2, 3])])
@pytest.mark.parametrize("N", [1, 100, 8191, 8193, 32767, 65536, 70001])
@pytest.mark.parametrize("dep", [0.0, 0.03])
def test_cluster_tests_match_oracle(F, arities, S, N, dep):
    import torch
    data, ar = _data(N, arities, dep)
    ref = oracle.ci_table(data, ar, 0, 1, S)
    for stat, df_mode in (("g2", "fixed"), ("x2", "adjusted")):
        h = F.fbn_create(data, ar, statistic=stat, df=df_mode)
        assert np.array_equal(F.fbn_ci_table(h, 0, 1, S), ref)
        g2, df, p = F.fbn_ci_test(h, 0, 1, S)
        rg2, rdf, rp = oracle.ci_test(data, ar, 0, 1, S, stat=stat, df_mode=df_mode)
        assert df == rdf and g2 == pytest.approx(rg2, rel=1e-6, abs=1e-12) and abs(p - rp) <= 1e-9
    ld = (N + 15) // 16 * 16
    dev = torch.zeros((len(ar), ld), dtype=torch.uint8, device="cuda")
    dev[:, :N] = torch.from_numpy(data).cuda()
    out = torch.zeros(3, dtype=torch.float64, device="cuda")
    table = torch.full((ref.size,), -7, dtype=torch.int32, device="cuda")
    F.fbn_ci_test_noalloc(dev, ld, N, ar, 0, 1, S, out, table)
    torch.cuda.synchronize()
    rg2, rdf, rp = oracle.ci_test(data, ar, 0, 1, S)
    assert out[1].item() == rdf and out[0].item() == pytest.approx(rg2, rel=1e-6, abs=1e-12)
    assert abs(out[2].item() - rp) <= 1e-9 and np.array_equal(table.cpu().numpy(), ref)


# One CTA (few samples, few cells): the warp that adds up the statistic and the one that
# prepares the p-value run side by side, so every repeat has to give the same bits.
@pytest.mark.parametrize("stat,df_mode", [("g2", "fixed"), ("g2", "adjusted"), ("x2", "fixed"), ("x2", "adjusted")])
def test_one_cta_repeats_bit_for_bit(F, stat, df_mode):
    data, ar = _data(3001, [2, 3, 2, 4], 0.05)
    h = F.fbn_create(data, ar, statistic=stat, df=df_mode)
    for S in ([], [2], [3, 2]):
        ref = oracle.ci_test(data, ar, 0, 1, S, stat=stat, df_mode=df_mode)
        first = F.fbn_ci_test(h, 0, 1, S)
        assert first[1] == ref[1] and first[0] == pytest.approx(ref[0], rel=1e-6) and abs(first[2] - ref[2]) <= 1e-9
        for _ in range(1000):
            assert F.fbn_ci_test(h, 0, 1, S) == first
