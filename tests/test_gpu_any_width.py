"""The any-width product kernel against the oracle: widths with and without a divisor that makes a
vector, wider than a warp's lanes, padded and misaligned blocks, off-centre sectors; and first products
of a process under capture, and beside one."""
import os
import subprocess
import sys

import numpy as np
import pytest

import workloads as wl
from oracle import hamiltonian as ham

from test_gpu_parity import _bound

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def mbl():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2012_00217_gb300 as m
    m.binding.lib()
    return m


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("L,n_up,periodic,k,ld,shift", [
    (12, 6, True, 20, 24, 0), (13, 4, False, 20, 20, 0), (11, 5, True, 33, 33, 0), (12, 6, False, 32, 33, 0),
    (10, 5, True, 64, 64, 1), (12, 5, True, 100, 104, 0), (9, 4, True, 256, 256, 0), (10, 5, False, 255, 255, 0),
    (14, 7, True, 6, 8, 2), (14, 7, False, 12, 12, 0), (4, 2, True, 5, 5, 0), (8, 0, True, 7, 7, 0),
    (16, 8, True, 1, 3, 0), (13, 13, False, 24, 24, 0), (5, 2, True, 31, 32, 0)])
def test_any_width(mbl, dtype, L, n_up, periodic, k, ld, shift):
    tdt = torch.float32 if dtype == np.float32 else torch.float64
    h = wl.fields(L, 6.0, 11 * L + k)
    chain = ham.Chain(L, h, delta=0.8, periodic=periodic, n_up=n_up)
    n = ham.sector_dim(L, n_up)
    Xb = wl.block(n, ld, 3 + k, dtype)
    ref = ham.apply(chain, 0.4, Xb[:, :k].astype(np.float64))
    xs = torch.empty(n * ld + shift, dtype=tdt, device=DEV)
    ys = torch.full((n * ld + shift,), 77.0, dtype=tdt, device=DEV)
    xs[shift:] = torch.from_numpy(Xb).to(DEV).flatten()
    X, Y = xs[shift:].view(n, ld)[:, :k], ys[shift:].view(n, ld)[:, :k]
    mbl.hamiltonian_apply(mbl.make_chain(L, h, 0.8, periodic, n_up), 0.4, X, Y)
    got = ys[shift:].view(n, ld).cpu().numpy()
    assert np.all(got[:, k:] == 77.0) and torch.all(ys[:shift] == 77.0)
    assert np.all(np.abs(got[:, :k].astype(np.float64) - ref) <= _bound(chain, 0.4, Xb[:, :k], dtype))


# A process whose first product of a tile width is captured (the any-width kernel's stand-in), or runs on
# another stream while one is being captured; torch captures in the mode that forbids the most
FIRST = """
import sys
import numpy as np, torch
import paper_2012_00217_gb300 as mbl
import workloads as wl
from oracle import hamiltonian as ham
L, k, beside = int(sys.argv[1]), int(sys.argv[2]), sys.argv[3] == "beside"
n = ham.sector_dim(L, L // 2)
h = wl.fields(L, 5.0, 1)
Xb = wl.block(n, k, 2)
ref = ham.apply(ham.Chain(L, h), 0.3, Xb)
chain = mbl.make_chain(L, h)
X = torch.from_numpy(Xb).cuda()
Y, Z = torch.zeros_like(X), torch.zeros_like(X)
other = torch.cuda.Stream()
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):
    if beside:
        with torch.cuda.stream(other):
            mbl.hamiltonian_apply(chain, 0.3, X, Z)
        Y.add_(X)
    else:
        mbl.hamiltonian_apply(chain, 0.3, X, Y)
other.synchronize()
for _ in range(2):
    Y.zero_()
    g.replay()
torch.cuda.synchronize()
assert np.abs((Z if beside else Y).cpu().numpy() - ref).max() <= 1e-11
if beside:
    assert torch.equal(X, Y)
print("agrees")
"""


@pytest.mark.parametrize("where", ["captured", "beside"])
@pytest.mark.parametrize("L,k", [(10, 20), (10, 32), (16, 20), (16, 32)])
def test_first_product_and_captures(mbl, L, k, where):
    r = subprocess.run([sys.executable, "-c", FIRST, str(L), str(k), where], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0 and "agrees" in r.stdout, r.stderr[-2000:]
