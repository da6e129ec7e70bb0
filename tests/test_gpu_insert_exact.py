"""Insertions keep their exact lists where the tiles cannot give them (GPU):
rows whose norms overflow FP32, and indexes made without tensor cores.

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
