"""The autotuner tunes the plain product: the order in which the resident PCG takes its work, and with it
the bits of a solve, stay what they were."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# in a process of its own: the tuner's choices stay for good
CODE = """
import torch, numpy as np
import paper_2012_00217_gb300 as mbl
import workloads as wl
from math import comb
def solve(ch, n, k):
    o = mbl.make_opts(4, k, tol=1e-14, max_iter=1, pcg_iters=20, norm_h=30.0, mode=1)
    ws = torch.empty(mbl.lobpcg_workspace_size(ch, o), dtype=torch.uint8, device="cuda")
    X0 = torch.randn(n, k, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    return mbl.lobpcg_solve(ch, 0.2, o, X0, ws, allow_not_converged=True)[0]
for L, n_up, k in ((24, 6, 32), (20, 9, 32), (19, 9, 64), (16, 8, 16)):
    n = comb(L, n_up)
    ch = mbl.make_chain(L, wl.fields(L, 6.0, 3), 1.0, True, n_up)
    before = solve(ch, n, k)
    X = torch.randn(n, k, dtype=torch.float32, device="cuda")
    choice = mbl.binding.autotune_product(ch, X, torch.empty_like(X), reps=5)
    assert np.array_equal(before, solve(ch, n, k)), (L, n_up, k, choice)
print("same bits")
"""


def test_autotuner_leaves_the_resident_pcg_alone():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0 and "same bits" in r.stdout, r.stderr[-2000:]
