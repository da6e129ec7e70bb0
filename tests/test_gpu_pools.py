"""Candidate pools of the distance tiles (GPU): exact k-NN, forward lists of
builds and insertions, at the edges of the tiles and of the pool, and on data
whose near ties send rows to the collecting pass or past its buffer.

Bound of a returned distance against FP64: each of the dpad / 32 FMA steps,
five butterfly additions, the subtraction (squared: twice) and the final square
root rounds by at most 2^-24, and rows scaled to unit length by a few more:
(dpad / 32 + 16) * 2^-23 relative covers them, taken against the largest
distance of the list where rows cancel (angular).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2505_17368_gb300")
torch = pytest.importorskip("torch")


def points(kind, n, d, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn(n, d, generator=g, device="cuda")
    if kind == "spread":
        return x
    # tight groups far from each other: the tile error of a pair, which goes
    # with the rows' norms, is as large as the distances within a group
    size = {"groups": 64, "crowds": 3000}[kind]
    centre = 30.0 * torch.randn((n + size - 1) // size, d, generator=g, device="cuda")
    which = torch.randperm(n, generator=g, device="cuda") // size
    return centre[which] + 0.02 * x


def truth(X, Q, k, metric):
    X, Q = X.double(), Q.double()
    if metric == H.ANGULAR:
        X, Q = X / X.norm(dim=1, keepdim=True), Q / Q.norm(dim=1, keepdim=True)
    out = []
    for q in Q.split(64):
        near = torch.cdist(q, X, compute_mode="donot_use_mm_for_euclid_dist").topk(k, largest=False, sorted=True).values
        out.append(0.5 * near * near if metric == H.ANGULAR else near)
    return torch.cat(out)


def check_dists(got, want, d, angular=False):
    rel = ((d + 31) // 32 + 16) * 2.0**-23
    # 1 - cos comes as half a squared distance of unit rows that are
    # themselves rounded: relative to 1 where the rows nearly agree
    tol = rel * want + (rel * want.clamp(min=1e-30).sqrt() * 4 + 2.0**-44 if angular else 0.0)
    assert (got.double() - want).abs().le(tol).all(), (got.double() - want).abs().max()


@pytest.mark.parametrize("kind", ["spread", "groups", "crowds"])
@pytest.mark.parametrize("n,d,nq,k,metric", [
    (8193, 32, 129, 10, H.L2), (65_536, 100, 17, 16, H.L2), (40_000, 128, 300, 17, H.L2), (20_001, 129, 64, 112, H.L2),
    (105, 24, 10_001, 112, H.L2), (255, 960, 5000, 1, H.L2), (30_000, 100, 128, 100, H.ANGULAR),
    (70_000, 16, 130, 48, H.ANGULAR)])
def test_exact_knn_against_fp64(kind, n, d, nq, k, metric):
    X = points(kind, n, d, 1)
    # near a row of the set, as far from it as its group is wide
    Q = X[torch.arange(nq, device="cuda") * 7919 % n] + 0.02 * points("spread", nq, d, 2)
    ids, dd = H.exact_knn(X, Q, k, metric=metric)
    kk = min(k, n)
    assert (ids[:, kk:] == -1).all() and torch.isinf(dd[:, kk:]).all()
    ids, dd = ids[:, :kk], dd[:, :kk]
    check_dists(dd, truth(X, Q, kk, metric), d, metric == H.ANGULAR)
    assert (dd[:, 1:] >= dd[:, :-1]).all()
    assert all(len(set(r)) == kk for r in ids.cpu().numpy().tolist())


@pytest.mark.parametrize("n,d,k,metric", [(3000, 40, 10, H.L2), (4000, 128, 100, H.L2), (4095, 72, 30, H.ANGULAR)])
def test_exact_knn_one_by_one_equals_batch(n, d, k, metric):
    """Few pairs take the SIMT path, many the tensor-core one: the same bits."""
    X, Q = points("spread", n, d, 3), points("spread", 512, d, 4)
    ids, dd = H.exact_knn(X, Q, k, metric=metric)
    for q in (0, 127, 128, 511):
        i1, d1 = H.exact_knn(X, Q[q:q + 1], k, metric=metric)
        assert torch.equal(i1[0], ids[q]) and torch.equal(d1[0], dd[q])


def test_exact_knn_not_finite():
    """With a point that is no number no list can be proven: every query takes the SIMT path, as one query does."""
    X, Q = points("spread", 4000, 48, 5), points("spread", 600, 48, 6)
    X = torch.cat([X, X[:1] * float("nan")])
    ids, dd = H.exact_knn(X, Q, 10)
    for q in (0, 599):
        i1, d1 = H.exact_knn(X, Q[q:q + 1], 10)
        assert torch.equal(i1[0], ids[q]) and torch.equal(d1[0].nan_to_num(-1.0), dd[q].nan_to_num(-1.0))


def test_exact_knn_in_a_graph():
    """Stream-ordered throughout: the call can be captured and replayed."""
    X, Q = points("groups", 20_000, 64, 7), points("groups", 200, 64, 8)
    want = H.exact_knn(X, Q, 20)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        H.exact_knn(X, Q, 20)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ids, dd = H.exact_knn(X, Q, 20)
        g.replay()
        s.synchronize()
    assert torch.equal(ids, want[0]) and torch.equal(dd, want[1])


@pytest.mark.parametrize("kind", ["spread", "groups", "crowds"])
@pytest.mark.parametrize("n,d,metric,graph", [
    (129, 32, H.L2, H.GRAPH_NSW), (5000, 100, H.L2, H.GRAPH_NSW), (12_345, 64, H.ANGULAR, H.GRAPH_NSW),
    (6000, 200, H.L2, H.GRAPH_NSW), (7001, 96, H.L2, H.GRAPH_KNN)])
def test_forward_lists_equal_the_simt_build(kind, n, d, metric, graph):
    X = points(kind, n, d, 9)
    a = H.Index(X, metric=metric, graph=graph, seed=3)
    b = H.Index(X, metric=metric, graph=graph, seed=3, tiles=H.TILES_SIMT)
    for i in range(len(a.info()["sizes"])):
        la, lb = a.layer(i), b.layer(i)
        for key in la:
            assert np.array_equal(la[key], lb[key]), (i, key)


@pytest.mark.parametrize("kind", ["spread", "groups", "crowds"])
@pytest.mark.parametrize("n,add,d,metric", [
    (4000, 1, 32, H.L2), (4000, 129, 100, H.L2), (9000, 1000, 72, H.ANGULAR), (3000, 300, 260, H.L2)])
def test_inserted_forward_lists(kind, n, add, d, metric):
    X = points(kind, n + add, d, 10)
    idx = H.Index(X[:n], metric=metric, seed=4)
    idx.insert(X[n:])
    fwd, fwd_d = (torch.from_numpy(idx.layer(0)[k][n:]).cuda() for k in ("fwd", "fwd_d"))
    Y = X.double()
    if metric == H.ANGULAR:
        Y = Y / Y.norm(dim=1, keepdim=True)
    for r in sorted({0, 1, add // 2, add - 1} & set(range(add))):
        dist = ((Y[:n + r] - Y[n + r]) ** 2).sum(1)
        if metric == H.ANGULAR:
            dist = 0.5 * dist
        check_dists(fwd_d[r], dist.topk(16, largest=False, sorted=True).values, d, metric == H.ANGULAR)
        assert len(set(fwd[r].tolist())) == 16


@pytest.mark.parametrize("graph", [H.GRAPH_NSW, H.GRAPH_KNN])
def test_open_rows_in_several_batches(graph):
    """More open rows than one collecting launch takes (128 per SM)."""
    X = points("groups", 45_000, 40, 11)
    a = H.Index(X, graph=graph, seed=3)
    b = H.Index(X, graph=graph, seed=3, tiles=H.TILES_SIMT)
    assert a.info()["uncertified_rows"] > 128 * torch.cuda.get_device_properties(0).multi_processor_count
    la, lb = a.layer(0), b.layer(0)
    assert all(np.array_equal(la[key], lb[key]) for key in la)
