"""Device memory of indexes (GPU): calls whose scratch does not fit."""
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
