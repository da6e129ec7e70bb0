"""Exact k-NN where the candidate lists prove nothing (GPU): batches whose near
ties overflow the collecting pass, calls too small for the tiles, and rows
whose norms overflow.  The
answer has to be the exact one there too, and the same for a query alone as
in a batch.
"""
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2505_17368_gb300")
torch = pytest.importorskip("torch")

from test_gpu_pools import check_dists, points, truth  # noqa: E402


def huge(n, d, seed, lead):
    """Finite rows on two sides of the origin, near ones 1e17 apart.  lead: "past" -- every squared norm overflows
    FP32; "around" -- about half of them do (the largest FP32 value is 1.8447e19 squared)."""
    x = 1e17 * points("spread", n, d, seed)
    side = torch.where(torch.arange(n, device="cuda") % 2 == 0, 1.0, -1.0)
    x[:, 0] = side * (2.2e19 if lead == "past" else 1.8447e19 + 0.1 * x[:, 0])
    return x


def near_rows(X, nq, seed):
    n, d = X.shape
    return X[torch.arange(nq, device="cuda") * 7919 % n] + 0.02 * points("spread", nq, d, seed)


# "crowds" of 3,000 points: with 10,000 queries one block of the collecting
# pass sees a whole crowd, more than it keeps for a query
@pytest.mark.parametrize("n,d,nq,k,metric", [
    (20_001, 32, 10_000, 10, H.L2), (20_000, 128, 9_999, 40, H.L2), (24_000, 100, 10_001, 112, H.ANGULAR)])
def test_batch_past_the_collecting_buffer(n, d, nq, k, metric):
    X = points("crowds", n, d, 21)
    Q = near_rows(X, nq, 22)
    ids, dd = H.exact_knn(X, Q, k, metric=metric)
    check_dists(dd, truth(X, Q, k, metric), d, metric == H.ANGULAR)
    assert (ids.sort(dim=1).values.diff(dim=1) > 0).all() and (ids >= 0).all()


@pytest.mark.parametrize("kind", ["spread", "groups", "crowds"])
@pytest.mark.parametrize("n,d,nq,k,metric", [
    (4095, 32, 1, 10, H.L2), (4000, 100, 1, 112, H.ANGULAR), (2047, 960, 2, 33, H.L2), (511, 7, 8, 64, H.L2),
    (1, 5, 3, 10, H.L2), (31, 128, 130, 65, H.ANGULAR)])
def test_small_calls_against_fp64(kind, n, d, nq, k, metric):
    X = points(kind, n, d, 23)
    Q = near_rows(X, nq, 24)
    ids, dd = H.exact_knn(X, Q, k, metric=metric)
    kk = min(k, n)
    assert (ids[:, kk:] == -1).all() and torch.isinf(dd[:, kk:]).all()
    check_dists(dd[:, :kk], truth(X, Q, kk, metric), d, metric == H.ANGULAR)
    assert all(len(set(r)) == kk for r in ids[:, :kk].cpu().numpy().tolist())


@pytest.mark.parametrize("kind", ["groups", "crowds"])
@pytest.mark.parametrize("n,d,k,metric", [(3000, 40, 10, H.L2), (4000, 128, 100, H.L2), (4095, 72, 30, H.ANGULAR)])
def test_one_by_one_equals_batch(kind, n, d, k, metric):
    X = points(kind, n, d, 25)
    Q = near_rows(X, 512, 26)
    ids, dd = H.exact_knn(X, Q, k, metric=metric)
    for q in (0, 127, 128, 511):
        i1, d1 = H.exact_knn(X, Q[q:q + 1], k, metric=metric)
        assert torch.equal(i1[0], ids[q]) and torch.equal(d1[0], dd[q])


@pytest.mark.parametrize("lead", ["past", "around"])
@pytest.mark.parametrize("n,d,nq,k", [(3000, 32, 500, 10), (2500, 200, 64, 100), (1200, 64, 2, 20)])
def test_norms_that_overflow(lead, n, d, nq, k):
    X = huge(n, d, 27, lead)
    Q = X[torch.arange(nq, device="cuda") * 7919 % n] * 1.001
    ids, dd = H.exact_knn(X, Q, k)
    check_dists(dd, truth(X, Q, k, H.L2), d)
    assert (ids >= 0).all() and (ids.sort(dim=1).values.diff(dim=1) > 0).all()
