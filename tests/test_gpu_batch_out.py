"""A batch's graphs into pageable, pinned and device memory in one call.

The pageable ones pass through a pinned buffer, 64 problems per launch, in
whole 16-byte words: odd variable counts, more problems than one launch takes
and skipped outputs between them.  Every graph equals the one learnt alone.
Separating sets read first through a member whose stream is not the batch's.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 64, 65, 131])
def test_batch_outputs(k):
    import torch
    import paper_2212_04259_gb300 as F
    rng = np.random.default_rng(k)
    hs, alone = [], []
    for p in range(k):
        n, N = int(rng.integers(2, 36)), int(rng.integers(100, 900))
        base = rng.integers(0, 3, N)
        x = np.stack([np.where(rng.random(N) < 0.5, base, rng.integers(0, 3, N)) for _ in range(n)]).astype(np.uint8)
        hs.append(F.fbn_create(x, np.full(n, 3, np.uint8)))
        alone.append(F.fbn_learn_skeleton(hs[-1], 0.05, 1))
    out = []
    for p, h in enumerate(hs):
        o = torch.full((h.n, h.n), 9, dtype=torch.uint8)
        out.append(o.numpy() if p % 3 == 0 else o.cuda() if p % 3 == 1 else o.pin_memory())
    F.fbn_learn_skeleton_batch(hs, 0.05, 1, adj_out=out)
    for p in range(k):
        got = out[p] if isinstance(out[p], np.ndarray) else out[p].cpu().numpy()
        assert np.array_equal(got, alone[p]), p
    for got, ref in zip(F.fbn_learn_skeleton_batch(hs, 0.05, 1), alone):
        assert np.array_equal(got, ref)


def test_sets_through_any_member():
    import torch
    import paper_2212_04259_gb300 as F
    rng = np.random.default_rng(1)
    hs, alone = [], []
    for n in (60, 40, 90, 30):
        base = rng.integers(0, 3, 600)
        x = np.stack([np.where(rng.random(600) < 0.45, base, rng.integers(0, 3, 600)) for _ in range(n)]).astype(np.uint8)
        hs.append(F.fbn_create(x, np.full(n, 3, np.uint8)))
        F.fbn_learn_skeleton(hs[-1], 0.01, 2)
        alone.append(F.fbn_export_sepsets(hs[-1]))
    streams = [torch.cuda.Stream() for _ in range(3)]
    for t in range(60):
        F.fbn_set_stream(hs[0], streams[t % 3])          # the pool changes streams between calls
        F.fbn_learn_skeleton_batch(hs, 0.01, 2)
        if t % 2:
            F.fbn_set_stream(hs[0], streams[(t + 1) % 3])
            F.fbn_learn_skeleton(hs[0], 0.01, 1)          # ... and is written again at once
        for q in (3, 1, 2) if t % 2 else (3, 0, 1, 2):
            assert F.fbn_export_sepsets(hs[q]) == alone[q], (t, q)
