"""Products on sectors with few (or nearly all) spins up on long chains, where nearly every tile is
empty: the values against the oracle, and the time against the untiled kernels, which go through
rows only."""
import math

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


def _time(mbl, chain, X, Y):
    g, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.stream(st):
        mbl.hamiltonian_apply(chain, 0.4, X, Y)
        g.capture_begin()
        for _ in range(5):
            mbl.hamiltonian_apply(chain, 0.4, X, Y)
        g.capture_end()
    best = float("inf")
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 200.0)
    return best


def _allowed(L, k, es, untiled):
    """Three times the untiled kernel and 20 us; for the widths of the tiled kernels also what their
    items without rows take at the largest chunks, 0.17 us each and warp (0.25 here), 24 warps an SM.
    With chunks sized by the rows alone these sectors took up to 650 us."""
    if k not in (1, 2, 4, 8, 16, 32, 64):
        return 3.0 * untiled + 20.0
    row, lane = k * es, 64 if es == 8 and k * es >= 128 else 32
    chunk = max(4 * (32 // max(1, row // lane)), 32)
    B = min(13, L - 2)
    items = 2 ** (L - B) * -(-math.comb(B, B // 2) // chunk)
    return 3.0 * untiled + 20.0 + 0.25 * items / (24 * torch.cuda.get_device_properties(0).multi_processor_count)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("L,n_up,periodic,k", [
    (28, 3, False, 64), (28, 2, True, 32), (28, 2, False, 8), (28, 3, True, 24), (28, 2, False, 20), (28, 1, True, 16),
    (28, 0, True, 20), (28, 27, True, 24), (28, 26, False, 8), (24, 22, True, 16), (22, 3, True, 32), (16, 15, True, 20),
    (12, 1, True, 1), (20, 17, True, 32)])
def test_sparse_sector(mbl, dtype, L, n_up, periodic, k):
    tdt = torch.float32 if dtype == np.float32 else torch.float64
    h = wl.fields(L, 6.0, L + k)
    chain = ham.Chain(L, h, delta=0.8, periodic=periodic, n_up=n_up)
    n = ham.sector_dim(L, n_up)
    Xb = wl.block(n, k, 3 + k, dtype)
    ref = ham.apply(chain, 0.4, Xb.astype(np.float64))
    X = torch.from_numpy(Xb).to(DEV)
    Y = torch.empty_like(X)
    mc = mbl.make_chain(L, h, 0.8, periodic, n_up)
    mbl.hamiltonian_apply(mc, 0.4, X, Y)
    assert np.all(np.abs(Y.cpu().numpy().astype(np.float64) - ref) <= _bound(chain, 0.4, Xb, dtype))
    us = _time(mbl, mc, X, Y)
    mbl.binding.set_product_tile_bits(k, tdt, -1)
    try:
        untiled = _time(mbl, mc, X, Y)
    finally:
        mbl.binding.set_product_tile_bits(k, tdt, 0)
    assert us <= _allowed(L, k, X.element_size(), untiled), (us, untiled)
