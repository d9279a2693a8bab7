"""The FP64 Jacobi eigensolver of the small matrices on graded ones, whose rotations have
(a_qq - a_pp) / (2 a_pq) up to 2^80 and beyond, against a plain FP64 Jacobi in numpy."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N = 32


@pytest.fixture(scope="module")
def small_eig():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2012_00217_gb300 as m
    fn = ctypes.CDLL(m.binding.LIB_PATH)["_ZN3mbl9small_eigEiPKdlPdS2_S2_P11CUstream_st"]
    fn.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_int64] + [ctypes.c_void_p] * 4
    w = torch.empty(N, dtype=torch.float64, device=DEV)
    Z = torch.empty(N, N, dtype=torch.float64, device=DEV)
    work = torch.empty(4 * N * (N + 1), dtype=torch.float64, device=DEV)

    def run(G):
        st = torch.cuda.current_stream().cuda_stream
        assert fn(N, G.data_ptr(), N, w.data_ptr(), Z.data_ptr(), work.data_ptr(), st) == 0
        return w, Z

    return run


def _graded(decades, seed):
    """D M D: M a Gram of condition about 10, D falling over `decades` decades in all."""
    rng = np.random.default_rng(seed)
    Q, _ = np.linalg.qr(rng.normal(size=(N, N)))
    M = (Q * np.linspace(1.0, 10.0, N)) @ Q.T
    D = 10.0 ** (-decades / 2 * np.arange(N) / (N - 1))
    return D[:, None] * (0.5 * (M + M.T)) * D[None, :]


def _jacobi(A):
    A = A.copy()
    for _ in range(30):
        rotated = False
        for p in range(N - 1):
            for q in range(p + 1, N):
                if abs(A[p, q]) <= 2.3e-16 * np.sqrt(abs(A[p, p] * A[q, q])):
                    continue
                rotated = True
                tau = (A[q, q] - A[p, p]) / (2.0 * A[p, q])
                t = np.copysign(1.0, tau) / (abs(tau) + np.hypot(1.0, tau))
                c = 1.0 / np.hypot(1.0, t)
                R = np.array([[c, t * c], [-t * c, c]])
                A[[p, q], :] = R.T @ A[[p, q], :]
                A[:, [p, q]] = A[:, [p, q]] @ R
                A[p, q] = A[q, p] = 0.0
        if not rotated:
            break
    return np.sort(np.diag(A))


# Demmel and Veselic: Jacobi's relative error on D M D is of the order n eps cond(M), 7e-14 here
@pytest.mark.parametrize("decades", [0, 14, 28, 45, 70])
def test_graded_relative_accuracy(small_eig, decades):
    G = _graded(decades, decades)
    want = _jacobi(G)
    w, Z = small_eig(torch.from_numpy(G).to(DEV))
    got, vec = w.cpu().numpy(), Z.cpu().numpy()
    assert np.all(np.abs(got - want) <= 3e-13 * want)
    assert np.abs(vec.T @ vec - np.eye(N)).max() <= 1e-13


@pytest.mark.parametrize("decades", [14, 28, 45])
def test_graded_sweeps_end(small_eig, decades):
    """A graded matrix takes no more sweeps than a full one (four to five against about eight); at
    the limit of 20 sweeps it would take more than twice the full one's time."""
    full = np.random.default_rng(1).normal(size=(N, N))
    mats = [torch.from_numpy(np.ascontiguousarray(G)).to(DEV) for G in (full + full.T, _graded(decades, 1))]
    best = [float("inf")] * 2
    for _ in range(15):
        for i, G in enumerate(mats):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            small_eig(G)
            b.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], a.elapsed_time(b))
    assert best[1] <= 1.3 * best[0], best
