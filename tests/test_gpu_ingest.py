"""New samples from every kind of memory, at every alignment.

The store, its check and the one-hot planes come from one pass over the
caller's rows: pinned host memory and device memory read in place (rows of any
length and buffers starting at any byte), pageable memory through a copy.
Tables and skeletons must be the oracle's, and a bad value is found in the
first, last and ragged words.
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


def _place(data, where, shift):
    """The samples in `where` memory, starting `shift` bytes into a buffer of
    values that would be refused."""
    import torch
    n, N = data.shape
    buf = torch.full((n * N + shift,), 255, dtype=torch.uint8)
    if where == "pinned":
        buf = buf.pin_memory()
    elif where == "device":
        buf = buf.cuda()
    out = buf[shift:].view(n, N)
    out.copy_(torch.from_numpy(data))
    return out


@pytest.mark.parametrize("where", ["pinned", "device", "pageable"])
@pytest.mark.parametrize("N", [1, 15, 31, 33, 255, 257, 8191, 8192, 8193, 16400])
def test_every_memory_and_alignment(F, where, N):
    rng = np.random.default_rng(N)
    ar = np.array([5, 2, 4, 3, 5], dtype=np.uint8)
    first = np.stack([rng.integers(0, r, N) for r in ar]).astype(np.uint8)
    h = F.fbn_create(_place(first, where, 3), ar)
    for shift in (0, 1, 2, 7, 13):
        data = np.stack([rng.integers(0, r, N) for r in ar]).astype(np.uint8)
        F.fbn_update_data_batch([h], [_place(data, where, shift)]) if shift & 1 else F.fbn_update_data(h, _place(data, where, shift))
        for x, y, S in ((0, 1, []), (2, 4, [3]), (4, 0, [2, 1])):
            assert np.array_equal(F.fbn_ci_table(h, x, y, S), oracle.ci_table(data, ar, x, y, S))
        ref = oracle.pc_stable(data, ar, 0.4, 1)   # depths 0 and 1 from the planes
        if not ref.near:
            assert np.array_equal(F.fbn_learn_skeleton(h, 0.4, 1), ref.adj)
    for v, smp in ((0, 0), (4, N - 1), (2, N // 2)):
        bad = first.copy()
        bad[v, smp] = ar[v]
        for call in (lambda: F.fbn_update_data(h, _place(bad, where, 5)),
                     lambda: F.fbn_update_data_batch([h], [_place(bad, where, 6)]),
                     lambda: F.fbn_create(_place(bad, where, 9), ar)):
            with pytest.raises(F.FbnError) as e:
                call()
            assert e.value.code == -2 and f"variable {v} at sample {smp} " in str(e.value)
        F.fbn_update_data(h, _place(first, where, 0))   # usable again
        assert np.array_equal(F.fbn_ci_table(h, 0, 1), oracle.ci_table(first, ar, 0, 1))


# The first bad value of a refused upload must not reach the next call, whatever its stream.
@pytest.mark.parametrize("where", ["pinned", "device"])
def test_refused_then_valid_repeatedly(F, where):
    import torch
    rng = np.random.default_rng(7)
    ar = np.array([3, 2, 4], dtype=np.uint8)
    good = np.stack([rng.integers(0, r, 4001) for r in ar]).astype(np.uint8)
    bad = good.copy()
    bad[1, 17] = 2
    good_m, bad_m = _place(good, where, 3), _place(bad, where, 3)
    h = F.fbn_create(good_m, ar)
    streams = [torch.cuda.Stream().cuda_stream, 0]
    for t in range(400):
        with pytest.raises(F.FbnError) as e:
            F.fbn_update_data(h, bad_m)
        assert "variable 1 at sample 17 " in str(e.value)
        if t % 3 == 0:
            F.fbn_set_stream(h, streams[t // 3 % 2])
        F.fbn_update_data(h, good_m)
    assert np.array_equal(F.fbn_ci_table(h, 2, 1, [0]), oracle.ci_table(good, ar, 2, 1, [0]))


# Only a part of the samples' memory is pinned: read through a copy, or refused by it, never in place.
@pytest.mark.parametrize("part", ["first", "last"])
def test_partly_pinned_samples(F, part):
    import torch
    rng = np.random.default_rng(3)
    ar = np.array([3, 2, 4, 5], dtype=np.uint8)
    N = 200_000
    buf = np.zeros(4 * N + 8192, np.uint8)
    at = -buf.ctypes.data % 4096
    data = buf[at:at + 4 * N].reshape(4, N)
    data[:] = np.stack([rng.integers(0, r, N) for r in ar])
    good = data.copy()
    h = F.fbn_create(good, ar)
    rt = torch.cuda.cudart()
    p = data.ctypes.data if part == "first" else data.ctypes.data + 4 * N // 4096 // 2 * 4096
    assert int(rt.cudaHostRegister(p, 2 * N // 4096 * 4096, 0)) == 0
    try:
        try:
            F.fbn_update_data(h, data)
        except F.FbnError as e:
            print("refused:", e)
            F.fbn_update_data(h, good)
        assert np.array_equal(F.fbn_ci_table(h, 0, 1, [2]), oracle.ci_table(good, ar, 0, 1, [2]))
        assert np.array_equal(F.fbn_ci_table(h, 3, 2, []), oracle.ci_table(good, ar, 3, 2, []))
    finally:
        assert int(rt.cudaHostUnregister(p)) == 0
