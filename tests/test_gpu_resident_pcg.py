"""The resident PCG kernel (all PCG steps of a lane in one cooperative launch): solves at the
edges of its splits against dense eigenvalues, and the batch's other place for w."""
import numpy as np
import pytest

import workloads as wl
from oracle import hamiltonian as ham

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


def _solve(mbl, L, n_up, h, periodic, sigma, nev, k, mode, norm_h, pcg_iters, pcg_tol=0.0):
    n = ham.sector_dim(L, n_up)
    chain = mbl.make_chain(L, h, 1.0, periodic, n_up)
    opts = mbl.make_opts(nev, k, tol=1e-8, max_iter=300, pcg_iters=pcg_iters, pcg_tol=pcg_tol, norm_h=norm_h, mode=mode)
    ws = torch.empty(mbl.lobpcg_workspace_size(chain, opts), dtype=torch.uint8, device=DEV)
    X0 = torch.from_numpy(wl.initial_block(n, k, 5)).to(DEV)
    return mbl.lobpcg_solve(chain, sigma, opts, X0, ws)


# one block of a lane (70 rows); a few; off-centre sectors; every width and both types; the
# 65th step, in a second launch; a freeze threshold.  Bounds: the method's, as elsewhere
@pytest.mark.parametrize("L,n_up,periodic,k,mode,pcg_iters,pcg_tol", [
    (8, 4, True, 8, 1, 30, 0.0), (8, 4, False, 8, 0, 30, 0.0), (10, 5, True, 16, 0, 65, 0.0),
    (12, 4, False, 16, 1, 65, 0.0), (12, 6, True, 32, 0, 40, 0.0), (13, 5, True, 32, 1, 129, 0.0),
    (12, 6, False, 64, 1, 20, 0.0), (11, 5, True, 64, 0, 20, 0.0), (13, 6, False, 8, 0, 64, 0.0),
    (12, 6, False, 16, 1, 200, 1e-3), (12, 6, False, 16, 0, 200, 1e-3)])
def test_solve_matches_dense(mbl, L, n_up, periodic, k, mode, pcg_iters, pcg_tol):
    h = wl.fields(L, 6.0, 40 + L)
    ev = np.linalg.eigvalsh(ham.dense_sector(ham.Chain(L, h, n_up=n_up, periodic=periodic)))
    sigma, norm_h = 0.5 * (ev[0] + ev[-1]), max(abs(ev[0]), abs(ev[-1]))
    nev = k // 2
    want = np.sort(ev[np.lexsort((ev, np.abs(ev - sigma)))[:nev]])
    evals, resid, stats, _ = _solve(mbl, L, n_up, h, periodic, sigma, nev, k, mode, norm_h, pcg_iters, pcg_tol)
    assert stats["converged"] == 1 and resid.max() <= 1e-8 * norm_h
    assert np.abs(evals - want).max() <= (1e-6 if mode else 1e-9) * norm_h
    again, _, _, _ = _solve(mbl, L, n_up, h, periodic, sigma, nev, k, mode, norm_h, pcg_iters, pcg_tol)
    assert np.array_equal(again, evals)  # every sum has a fixed order


# whole tiles through shared memory, by the switch: every width and type, rows below 128 bytes (whose
# records stay in global memory) and above, more tiles than the groups have cached jobs for, one block
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("L,n_up,periodic,k,nev", [
    (12, 6, True, 8, 4), (13, 5, False, 8, 4), (12, 6, False, 16, 8), (12, 6, True, 32, 16), (12, 7, False, 64, 32),
    (8, 4, True, 16, 8), (14, 7, False, 64, 16)])
def test_staged_solve_matches_dense(mbl, L, n_up, periodic, k, nev, mode):
    h = wl.fields(L, 6.0, 80 + L)
    ev = np.linalg.eigvalsh(ham.dense_sector(ham.Chain(L, h, n_up=n_up, periodic=periodic)))
    sigma, norm_h = 0.5 * (ev[0] + ev[-1]), max(abs(ev[0]), abs(ev[-1]))
    want = np.sort(ev[np.lexsort((ev, np.abs(ev - sigma)))[:nev]])
    try:
        for t in (torch.float32, torch.float64):
            mbl.binding.set_product_schedule(k, t, 3)
        evals, resid, stats, _ = _solve(mbl, L, n_up, h, periodic, sigma, nev, k, mode, norm_h, 40)
        again, _, _, _ = _solve(mbl, L, n_up, h, periodic, sigma, nev, k, mode, norm_h, 40)
    finally:
        for t in (torch.float32, torch.float64):
            mbl.binding.set_product_schedule(k, t, 0)
    assert stats["converged"] == 1 and resid.max() <= 1e-8 * norm_h
    assert np.abs(evals - want).max() <= (1e-6 if mode else 1e-9) * norm_h
    assert np.array_equal(again, evals)


def test_batch_with_w_outside_tensor_memory(mbl):
    """64 lanes on the SMs leave a lane of 3,432 rows two blocks, 1,716 rows each: more than the
    1,008 rows of 32 FP64 columns that a block's tensor memory holds.  The single solve (23
    rows a block) keeps w there; both converge to the same eigenvalues."""
    L, k, nev, nprob = 14, 32, 4, 64
    hs = [wl.batched_fields(L, 8.0, s) for s in range(nprob)]
    chains = [mbl.make_chain(L, h) for h in hs]
    n = ham.sector_dim(L, 7)
    sigmas = [0.1] * nprob
    opts = mbl.make_opts(nev, k, tol=1e-8, max_iter=100, pcg_iters=66, norm_h=30.0, mode=0)
    ws = torch.empty(mbl.binding.batched_workspace_size(chains, opts, nprob), dtype=torch.uint8, device=DEV)
    X0 = torch.from_numpy(np.concatenate([wl.initial_block(n, k, s) for s in range(nprob)])).to(DEV)
    evals, resid, stats, _ = mbl.binding.lobpcg_solve_batched(chains, opts, X0, ws, nprob, sigmas=sigmas)
    assert all(s["converged"] for s in stats) and resid.max() <= 1e-8 * 30.0
    one = torch.empty(mbl.lobpcg_workspace_size(chains[0], opts), dtype=torch.uint8, device=DEV)
    for i in (0, 31, 63):
        single, _, _, _ = mbl.lobpcg_solve(chains[i], sigmas[i], opts, X0[i * n:(i + 1) * n].contiguous(), one)
        assert np.abs(single - evals[i]).max() <= 1e-9 * 30.0


# the resident Lanczos kernel: one block, several, off-centre sectors, an invariant subspace
# (n_up = 1: it ends at step n), a last launch of fewer steps.  1e-9: the residual bound of the
# call, 1e-7 relative, squared over a gap of the spectrum's ends
@pytest.mark.parametrize("L,n_up,periodic,max_iter", [
    (4, 2, True, 400), (6, 3, False, 400), (9, 1, True, 9), (10, 4, True, 400), (12, 6, False, 133), (13, 5, True, 400)])
def test_resident_lanczos_matches_dense(mbl, L, n_up, periodic, max_iter):
    h = wl.fields(L, 5.0, 60 + L)
    ev = np.linalg.eigvalsh(ham.dense_sector(ham.Chain(L, h, n_up=n_up, periodic=periodic)))
    chain = mbl.make_chain(L, h, 1.0, periodic, n_up)
    n = ham.sector_dim(L, n_up)
    X0 = torch.from_numpy(wl.block(n, 2, 8)).to(DEV)
    ws = torch.empty(mbl.bounds_workspace_size(chain, 2), dtype=torch.uint8, device=DEV)
    lo, hi, steps = mbl.spectrum_bounds(chain, X0, ws, tol=1e-7, max_iter=max_iter)
    scale = max(abs(ev[0]), abs(ev[-1]))
    assert abs(lo - ev[0]) <= 1e-9 * scale and abs(hi - ev[-1]) <= 1e-9 * scale and 1 <= steps <= max_iter
    assert mbl.spectrum_bounds(chain, X0, ws, tol=1e-7, max_iter=max_iter) == (lo, hi, steps)
