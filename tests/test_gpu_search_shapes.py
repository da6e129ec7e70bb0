"""Launch shapes of the search (GPU): the rows in flight, the warps per block
and the long lists' insertion follow the number of queries and the beam width,
and must not change an answer; ring distances for every number of ranges; the
device pool under several threads.
"""
import gc
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


@pytest.mark.parametrize("storage", [H.F32, H.BF16, H.FP8E4M3])
@pytest.mark.parametrize("d", [20, 64, 128, 500, 1000])
def test_answers_do_not_depend_on_the_launch(storage, d):
    """A full launch (4,500 queries), one of 14 warps per SM, one of a few per SM and single queries."""
    X, Q = rand(6000, d, 1), rand(4500, d, 2)
    idx = H.Index(X, storage=storage, seed=1)
    keys = torch.arange(4500, device="cuda", dtype=torch.int64)
    for ef in (10, 64, 65, 97, 300):
        for kw in (dict(ef_upper=1), dict(ef_upper=40, descend_all=1)):
            ids, dd, _ = idx.search(Q, k=10, ef=ef, keys=keys, warps_per_block=4, **kw)
            for a, b in ((0, 2000), (100, 1000), (7, 8), (4499, 4500)):
                i1, d1, _ = idx.search(Q[a:b], k=10, ef=ef, keys=keys[a:b], **kw)
                assert torch.equal(i1, ids[a:b]) and torch.equal(d1, dd[a:b]), (ef, kw, a, b)


def test_long_beam_keeps_every_point_it_reaches():
    """A beam as wide as the set ends with every reachable point once, in order: each insertion into its list counts."""
    X, Q = rand(700, 24, 3), rand(40, 24, 4)
    idx = H.Index(X, seed=2)
    base = idx.layer(0)
    adj = base["adj"]
    # every point's first link leads towards the first inserted one (which
    # has none forward); links are one-way: a point need not be in any row
    root = int(np.nonzero(base["fwd"][:, 0] < 0)[0][0])
    reached, todo = {root}, [root]
    while todo:
        for v in adj[todo.pop()].tolist():
            if v >= 0 and v not in reached:
                reached.add(v)
                todo.append(v)
    ids, dd, _ = idx.search(Q, k=700, ef=700)
    for q in range(40):
        got = ids[q][ids[q] >= 0]
        dist = dd[q, :len(got)]
        assert reached <= set(got.tolist()) and len(set(got.tolist())) == len(got)
        want = (X[got].double() - Q[q].double()).norm(dim=1)
        assert (dist.double() - want).abs().max() <= 16 * 2.0**-23 * want.max()
        assert (dist[1:] >= dist[:-1]).all() and torch.isinf(dd[q, len(got):]).all()


@pytest.mark.parametrize("metric", [H.L2, H.ANGULAR])
@pytest.mark.parametrize("ranges", [1, 32, 33, 64, 65, 104, 105, 211])
def test_layers_for_every_number_of_ranges(ranges, metric):
    import oracle as O

    X = rand(5003, 9, 5).cpu().numpy()
    g = H.Index(X, seed=6, num_ranges=ranges, eps_c0=0.3, metric=metric)
    o = O.build_layers(X, seed=6, r=ranges, c0=0.3, metric=metric)
    assert g.info()["sizes"] == [len(a) for a in o["ids"]]
    for i in range(1, len(o["ids"])):
        assert np.array_equal(g.layer(i)["ids"], o["ids"][i])


def test_builds_in_threads_share_the_pool():
    """Builds, insertions and frees in four threads, each on its own stream; the graphs are read once all have ended."""
    X = [rand(4000 + 700 * t, 48, 10 + t) for t in range(4)]
    want = []
    for x in X:
        idx = H.Index(x[:-50], seed=7)
        idx.insert(x[-50:])
        want.append(idx.layer(0))
    del idx
    last, failed = [None] * 4, []

    def work(t):
        try:
            for _ in range(6):
                stream = torch.cuda.Stream()
                idx = H.Index(X[t][:-50], seed=7, stream=stream)
                idx.insert(X[t][-50:], stream=stream)
                if last[t] is not None:
                    last[t].close()
                last[t] = idx
        except Exception as e:  # reported below
            failed.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for t in range(4):
        got = last[t].layer(0)
        assert all(np.array_equal(got[k], want[t][k]) for k in got)


def test_freed_indexes_give_their_memory_back():
    gc.collect()
    idx = H.Index(rand(400_000, 128, 20), storage=H.BF16, seed=8)
    torch.cuda.empty_cache()
    held = idx.info()["device_bytes"]
    before = torch.cuda.mem_get_info()[0]
    idx.close()
    # all but what the pool keeps once the last index is gone
    assert torch.cuda.mem_get_info()[0] - before >= held - (256 << 20) - (32 << 20)


@pytest.mark.parametrize("storage,d", [(H.F32, 100), (H.BF16, 64), (H.FP8E4M3, 400)])
def test_searches_side_by_side(storage, d):
    """The launches of several streams choose their kernels by one another; the answers are those of one stream."""
    X, Q = rand(8000, d, 21), rand(6 * 700, d, 22)
    idx = H.Index(X, storage=storage, seed=9)
    keys = torch.arange(len(Q), device="cuda", dtype=torch.int64)
    want = idx.search(Q, k=10, ef=64, keys=keys)[:2]
    torch.cuda.synchronize()
    failed = []

    def work(t):
        try:
            stream = torch.cuda.Stream()
            part = slice(700 * t, 700 * (t + 1))
            out = [idx.search(Q[part], k=10, ef=64, keys=keys[part], stream=stream) for _ in range(12)]
            stream.synchronize()
            for ids, dd, _ in out:
                assert torch.equal(ids, want[0][part]) and torch.equal(dd, want[1][part])
        except Exception as e:  # reported below
            failed.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
