"""Where the blocks of a cooperative launch do not fit (a context that has a part of the SMs), bounds,
solves and batches take the launches that wait for nothing.  The failing call is replaced on the host:
the library is linked once more with a cooperative_launch that always answers kTooLarge."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = """
#include "mbl_internal.h"
namespace mbl {
int cooperative_launch(const void *, unsigned, unsigned, size_t, void **, cudaStream_t) { return kTooLarge; }
}
"""

CODE = """
import sys
import numpy as np, torch
import paper_2012_00217_gb300 as mbl
import workloads as wl
from oracle import hamiltonian as ham
if sys.argv[1:]:
    mbl.binding.LIB_PATH = sys.argv[1]
L, k, nev = 12, 16, 8
n = ham.sector_dim(L, 6)
h = wl.fields(L, 6.0, 2)
ev = np.linalg.eigvalsh(ham.dense_sector(ham.Chain(L, h, n_up=6)))
chain = mbl.make_chain(L, h)
X0 = torch.from_numpy(wl.initial_block(n, k, 5)).cuda()
ws = torch.empty(mbl.bounds_workspace_size(chain, 4), dtype=torch.uint8, device="cuda")
lo, hi, steps = mbl.spectrum_bounds(chain, X0[:, :4].contiguous(), ws, tol=1e-7, max_iter=300)
scale = max(abs(ev[0]), abs(ev[-1]))
assert abs(lo - ev[0]) <= 1e-9 * scale and abs(hi - ev[-1]) <= 1e-9 * scale
sigma = 0.5 * (lo + hi)
want = np.sort(ev[np.argsort(np.abs(ev - sigma))[:nev]])
for graph in (0, 1):
    for mode in (0, 1):
        o = mbl.make_opts(nev, k, tol=1e-8, max_iter=200, pcg_iters=70, norm_h=scale, mode=mode, use_graph=graph)
        w = torch.empty(mbl.lobpcg_workspace_size(chain, o), dtype=torch.uint8, device="cuda")
        got, resid, st, _ = mbl.lobpcg_solve(chain, sigma, o, X0, w)
        assert st["converged"] and np.abs(np.sort(got) - want).max() <= (1e-6 if mode else 1e-9) * scale
    chains = [chain] * 3
    w = torch.empty(mbl.binding.batched_workspace_size(chains, o, 2), dtype=torch.uint8, device="cuda")
    got, resid, st, _ = mbl.binding.lobpcg_solve_batched(chains, o, X0.repeat(3, 1), w, 2)
    assert all(s["converged"] for s in st) and np.abs(np.sort(got, axis=1) - want).max() <= 1e-6 * scale
print("agrees")
"""


def test_without_cooperative_launches(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_00217_gb300 import build
    src, obj, so = tmp_path / "fake.cu", str(tmp_path / "fake.o"), str(tmp_path / "libmbl_no_coop.so")
    src.write_text(FAKE)
    subprocess.run([build.NVCC] + build.FLAGS + ["-c", str(src), "-o", obj], check=True)
    objs = [os.path.join(build.BUILD_DIR, s[:-3] + ".o") for s in build.SOURCES if s != "mbl_coop.cu"]
    subprocess.run([build.NVCC, "-shared", "-gencode", "arch=compute_103a,code=sm_103a", "-o", so] + objs + [obj], check=True)
    for args in ([], [so]):
        r = subprocess.run([sys.executable, "-c", CODE] + args, capture_output=True, text=True, timeout=300, cwd=ROOT)
        assert r.returncode == 0 and "agrees" in r.stdout, (args, r.stderr[-2000:])
