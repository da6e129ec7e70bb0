"""Insertions keep their exact lists where the tiles cannot give them (GPU):
rows whose norms overflow FP32.
"""
import pytest

pytestmark = pytest.mark.gpu

H = pytest.importorskip("paper_2505_17368_gb300")
torch = pytest.importorskip("torch")

from test_gpu_knn_exact import huge  # noqa: E402
from test_gpu_pools import check_dists  # noqa: E402


@pytest.mark.parametrize("lead", ["past", "around"])
@pytest.mark.parametrize("n,add,d", [(2000, 60, 32), (1500, 300, 200)])
def test_inserted_rows_whose_norms_overflow(lead, n, add, d):
    X = huge(n + add, d, 31, lead)
    idx = H.Index(X[:n], seed=4)
    idx.insert(X[n:])
    fwd, fwd_d = (torch.from_numpy(idx.layer(0)[k][n:]).cuda() for k in ("fwd", "fwd_d"))
    Y = X.double()
    for r in sorted({0, 1, add // 2, add - 1}):
        want = ((Y[:n + r] - Y[n + r]) ** 2).sum(1).topk(16, largest=False, sorted=True).values
        check_dists(fwd_d[r], want, d)
        assert len(set(fwd[r].tolist())) == 16 and (fwd[r] >= 0).all()
