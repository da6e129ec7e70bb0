"""Device memory of indexes (GPU): calls whose scratch does not fit, and freeing
with searches in flight, on a full device and beside a capture, and deletion
on a capturing stream."""
import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2505_17368_gb300")
torch = pytest.importorskip("torch")


def rand(n, d, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(n, d, generator=g, device="cuda")


def test_insertion_into_a_full_device():
    """With 300 MB left, the tiles' scratch (0.9 GB) does not fit: the rows are scanned, with the same lists."""
    X = rand(440_000, 512, 1)
    a, b = (H.Index(X, storage=H.BF16, seed=3) for _ in range(2))
    new = rand(200, 512, 2).cpu().numpy()
    del X
    for idx in (a, b):
        idx.insert(new[:100])  # the arrays grow
    torch.cuda.empty_cache()
    full = torch.empty(torch.cuda.mem_get_info()[0] - (300 << 20), dtype=torch.uint8, device="cuda")
    a.insert(new[100:])
    del full
    torch.cuda.empty_cache()
    b.insert(new[100:])
    la, lb = a.layer(0), b.layer(0)
    assert all(np.array_equal(la[key], lb[key]) for key in la)
    for x, y in zip(a.search(new, k=10, ef=64), b.search(new, k=10, ef=64)):
        assert np.array_equal(x, y)


def searches_in_flight(idx, Q, stream):
    """Enough of them that the stream is still busy when this returns."""
    with torch.cuda.stream(stream):
        out = [idx.search(Q, k=10, ef=512, ef_upper=32, stream=stream)[:2] for _ in range(40)]
    assert not stream.query()
    return out


def test_close_waits_for_searches_in_flight():
    X, Q = rand(100_000, 64, 4), rand(10_000, 64, 5)
    idx, other = H.Index(X, seed=1), H.Index(X[:1000], seed=1)
    want = idx.search(Q, k=10, ef=512, ef_upper=32)[:2]
    stream = torch.cuda.Stream()
    out = searches_in_flight(idx, Q, stream)
    idx.close()
    assert stream.query()
    other.close()
    for ids, dd in out:
        assert torch.equal(ids, want[0]) and torch.equal(dd, want[1])


def test_close_on_a_full_device():
    """Not a byte left to allocate: freeing waits all the same."""
    X, Q = rand(100_000, 64, 4), rand(10_000, 64, 5)
    idx = H.Index(X, seed=1)
    want = idx.search(Q, k=10, ef=512, ef_upper=32)[:2]
    stream = torch.cuda.Stream()
    out = searches_in_flight(idx, Q, stream)  # (their buffers come first)
    torch.cuda.synchronize()
    del out
    cudart = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    held, size = [], 1 << 36
    out = searches_in_flight(idx, Q, stream)
    while size >= 512:
        p = ctypes.c_void_p()
        if cudart.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0:
            held.append(p)
        else:
            size //= 2
    cudart.cudaGetLastError()
    try:
        idx.close()
        assert stream.query()
    finally:
        for p in held:
            cudart.cudaFree(p)
    for ids, dd in out:
        assert torch.equal(ids, want[0]) and torch.equal(dd, want[1])


@pytest.mark.parametrize("other_thread", [False, True])
def test_close_beside_a_capture(other_thread):
    """A capture in progress, in the default mode that other threads' calls can spoil, stays whole."""
    X = rand(3000, 32, 6)
    idx = H.Index(X, seed=1)
    idx.search(X[:100], k=10)
    g, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    y = torch.zeros_like(X)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        y.copy_(X)
        y.mul_(2.0)
        if other_thread:
            t = threading.Thread(target=idx.close)
            t.start()
            t.join()
        else:
            idx.close()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, 2.0 * X)


def test_threads_close_searched_indexes_beside_builds():
    """Builds capture their steps; another thread's close must not spoil them."""
    X = [rand(4000 + 300 * t, 48, 10 + t) for t in range(4)]
    indexes = [H.Index(x, seed=2) for x in X]
    want = [idx.search(x[:200], k=10)[0] for x, idx in zip(X, indexes)]
    torch.cuda.synchronize()
    failed = []

    def work(t):
        try:
            stream = torch.cuda.Stream()
            for _ in range(8):
                idx = H.Index(X[t], seed=2, stream=stream)
                got = idx.search(X[t][:200], k=10, stream=stream)  # all of it kept until the stream is done
                idx.close()
                stream.synchronize()
                assert torch.equal(got[0], want[t])
        except Exception as e:  # reported below
            failed.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed


def test_delete_on_a_capturing_stream_is_refused():
    """Before anything has changed: the index searches on, and the capture stays whole."""
    X = rand(3000, 32, 7)
    idx = H.Index(X, seed=1)
    want = idx.search(X[:100], k=10)[0]
    g, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    y = torch.zeros_like(X)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=stream):
        y.copy_(X)
        with pytest.raises(H.HennError):
            idx.delete([0, 1, 2], stream=stream)
    g.replay()
    assert torch.equal(idx.search(X[:100], k=10)[0], want)
    idx.delete([0, 1, 2])
    got = idx.search(X[:100], k=10)[0]
    assert not torch.isin(got, torch.arange(3, device="cuda")).any() and torch.equal(y, X)


def test_insertion_that_runs_out_of_memory():
    """Whichever array does not fit any more, the index answers as before and takes the rows once there is room."""
    X, new = rand(300_000, 512, 8), rand(20_000, 512, 9).cpu().numpy()
    Q = X[:500] + 0.01
    want = H.Index(X, storage=H.BF16, seed=3)
    want.insert(new)
    want = want.layer(0)
    refused = 0
    for left in (100, 1300, 1400, 1600, 2000, 2600):
        idx = H.Index(X, storage=H.BF16, seed=3)
        before = [t.clone() for t in idx.search(Q, k=10)[:2]]
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        full = torch.empty(torch.cuda.mem_get_info()[0] - (left << 20), dtype=torch.uint8, device="cuda")
        try:
            idx.insert(new)
        except H.HennError as e:
            assert e.status == 2
            refused += 1
        del full
        torch.cuda.empty_cache()
        if idx.n == 300_000:
            assert all(torch.equal(a, b) for a, b in zip(idx.search(Q, k=10)[:2], before))
            idx.insert(new)
        got = idx.layer(0)
        assert all(np.array_equal(got[key], want[key]) for key in want)
        idx.close()
    assert refused >= 1


def test_scratch_is_kept_beside_large_indexes():
    """An index of over 1 GiB: its insertions' scratch (0.9 GB) stays in the pool between calls, and goes with it."""
    idx = H.Index(rand(440_000, 512, 1), storage=H.BF16, seed=3)
    new = rand(100, 512, 2).cpu().numpy()
    idx.insert(new)  # the arrays have doubled: 880,000 rows
    arrays = 880_000 * (512 * 6 + 32 * 4 + 16 * 8)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    idx.close()
    back = torch.cuda.mem_get_info()[0] - before
    # all but what the pool keeps once the last index is gone; the upper layers' arrays come on top
    assert arrays + 850e6 - (256 << 20) <= back <= 1.1 * arrays + (1 << 30)


def test_deletion_whose_rebuild_runs_out_of_memory():
    """The upper layers go, the index answers from what is left, without the deleted points."""
    X = rand(3_000_000, 16, 12)
    idx = H.Index(X, storage=H.BF16, seed=5)
    upper = idx.layer(1)["ids"]
    gone = np.concatenate([upper[: 2 * len(upper) // 3], np.arange(0, 3_000_000, 1000)])
    Q = X[:300].cpu().numpy()
    idx.search(Q, k=10, ef=128)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    # the rings of layer 1 want 1.2 GB, the pool keeps 1 GiB at most
    full = torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")
    with pytest.raises(H.HennError) as e:
        idx.delete(gone)
    assert e.value.status == 2
    assert len(idx.info()["sizes"]) == 1 and idx.info()["L"] == 0
    ids = idx.search(Q, k=10, ef=128)[0]
    del full
    dead = np.zeros(3_000_000, bool)
    dead[gone] = True
    assert (ids >= 0).all() and not dead[ids].any()
    assert np.array_equal(idx.search(Q, k=10, ef=128)[0], ids)
    idx.delete(np.arange(5, 100_000, 7))
    again = idx.search(Q, k=10, ef=128)[0]
    assert (again >= 0).all() and not (again % 7 == 5)[again < 100_000].any()
