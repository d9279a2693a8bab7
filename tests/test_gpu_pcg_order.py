"""The PCG steps of a solve, resident and beyond L2, in sectors on and off the middle: the default work
order against the two it chooses from."""
import pytest

import workloads as wl
from oracle import hamiltonian as ham

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("L,n_up,k,mode", [(24, 7, 64, 1), (23, 8, 32, 1), (22, 9, 64, 1), (22, 11, 32, 1), (22, 7, 32, 0),
                                           (22, 10, 32, 0), (20, 10, 32, 0), (23, 8, 16, 0),
                                           (20, 10, 32, 1), (20, 9, 32, 1), (19, 9, 64, 1), (21, 10, 16, 1), (24, 6, 32, 1),
                                           (22, 7, 32, 1), (20, 9, 16, 0), (18, 9, 64, 0)])
def test_pcg_order(L, n_up, k, mode):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2012_00217_gb300 as mbl
    n = ham.sector_dim(L, n_up)
    chain = mbl.make_chain(L, wl.fields(L, 8.0, 1), 1.0, True, n_up)
    opts = mbl.make_opts(8, k, tol=1e-14, max_iter=1, pcg_iters=30, norm_h=40.0, mode=mode, use_graph=0, timing=1)
    ws = torch.empty(mbl.lobpcg_workspace_size(chain, opts), dtype=torch.uint8, device=DEV)
    X0 = torch.randn(n, k, dtype=torch.float64, device=DEV)
    types = (torch.float32, torch.float64)
    us = []
    try:
        for order in (0, 1, 3):
            for t in types:
                mbl.binding.set_product_schedule(k, t, order)
            us.append(min(mbl.lobpcg_solve(chain, -1.8, opts, X0, ws, allow_not_converged=True)[2]["t_pcg"]
                          for _ in range(5)) / 30 * 1e6)
    finally:
        for t in types:
            mbl.binding.set_product_schedule(k, t, 0)
    assert us[0] <= 1.08 * min(us[1:]), us
