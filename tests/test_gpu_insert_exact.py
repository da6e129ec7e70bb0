"""Insertions keep their exact lists where the tiles cannot give them (GPU):
rows whose norms overflow FP32, indexes made without tensor cores, and tile
launches that time out; so do open rows of builds and exact k-NN.

The tile pipeline is held by environment switches (its loads are not issued
and its bounded waits run out), in a child process that no other test shares.
"""
import os
import subprocess
import sys

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


CHILD = r"""
import os, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import paper_2505_17368_gb300 as H
import synth

def held(on):
    for key, value in (("HENN_TILE_HOLD_LOADS", on), ("HENN_TILE_SPIN_LIMIT", "256")):
        if on:
            os.environ[key] = value
        else:
            os.environ.pop(key, None)

def same(a, b):
    for i in range(len(a.info()["sizes"])):
        la, lb = a.layer(i), b.layer(i)
        assert all(np.array_equal(la[k], lb[k]) for k in la), i

X = synth.uniform_cube(5200, 48, seed=5)
"""


def run_child(code):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD + code, root], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr[-3000:]


def test_simt_index_inserts_without_tensor_cores():
    run_child("""
want = H.Index(X[:5000], seed=2)
want.insert(X[5000:])
idx = H.Index(X[:5000], seed=2, tiles=H.TILES_SIMT)
held("1")
idx.insert(X[5000:])
held("")
same(idx, want)
print("ok")
""")


def test_insertion_whose_tiles_time_out():
    """The new rows are scanned; the index, whose arrays have grown, goes on."""
    run_child("""
want = H.Index(X[:5000], seed=2)
want.insert(X[5000:])
idx = H.Index(X[:5000], seed=2)
held("1")
idx.insert(X[5000:])
held("")
same(idx, want)
assert idx.search(X[5000:], k=1, ef=64)[0][:, 0].tolist() == list(range(5000, 5200))
idx.insert(X[:300])
want.insert(X[:300])
same(idx, want)
print("ok")
""")


def test_collecting_passes_that_time_out():
    """Tight groups far apart leave rows open; with only the collecting launches held these are scanned."""
    run_child("""
g = np.random.default_rng(3)
X = (30.0 * g.standard_normal((90, 48)))[g.integers(90, size=6000)] + 0.02 * g.standard_normal((6000, 48))
X = X.astype(np.float32)
want = H.Index(X[:5800], seed=2)
assert want.info()["uncertified_rows"] > 0
held("2")
idx = H.Index(X[:5800], seed=2)
same(idx, want)
idx.insert(X[5800:])
held("")
want.insert(X[5800:])
same(idx, want)
print("ok")
""")


def test_exact_knn_whose_tiles_time_out():
    run_child("""
import torch
X = torch.from_numpy(X).cuda()
for k in (10, 60):
    want = H.exact_knn(X, X[:700] + 0.01, k)
    for hold in "12":
        held(hold)
        got = H.exact_knn(X, X[:700] + 0.01, k)
        held("")
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]), (k, hold)
print("ok")
""")
