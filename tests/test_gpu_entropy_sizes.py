"""Entanglement entropy at the edges of its kernels' splits, against the oracle's SVD: Gram sides
of 1 to 70 around a warp and a tile, unequal sides, graded spectra (localized vectors), degenerate
spectra, and the sizes whose rows do and do not fit in shared memory (252 and 462)."""
import math

import numpy as np
import pytest

from oracle import hamiltonian as ham
from oracle import observables as obs

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


def _columns(L, st, rng):
    peak = st[rng.integers(st.size)]
    dist = np.array([bin(int(s) ^ int(peak)).count("1") for s in st])
    V = rng.normal(size=(st.size, 4))
    V[:, 1] *= np.exp(-1.8 * dist)      # singular values over 20 orders of magnitude
    V[:, 2] = (dist <= 2) * 1.0         # many equal and zero singular values
    V[:, 3] = np.exp(-40.0 * dist)      # all but one below rounding
    return V


# |S - oracle| <= 1e-10: the bound of the other entropy tests
@pytest.mark.parametrize("L,n_up,l_a", [(2, 1, 1), (6, 3, 3), (9, 4, 2), (12, 5, 7), (14, 7, 6), (15, 7, 8), (16, 8, 8),
                                        (16, 0, 8), (16, 16, 4), (20, 10, 10), (20, 8, 13), (22, 11, 11)])
def test_entropy_sizes(mbl, L, n_up, l_a):
    rng = np.random.default_rng(L * 31 + l_a)
    st = ham.basis(L, n_up)
    V = _columns(L, st, rng)[:, :4 if L < 22 else 2]
    chain = mbl.make_chain(L, np.zeros(L), 1.0, False, n_up)
    S = mbl.entanglement_entropy(chain, l_a, torch.from_numpy(V.copy()).to(DEV)).cpu().numpy()
    for e in range(V.shape[1]):
        assert abs(S[e] - obs.entanglement_entropy(st, V[:, e], l_a)) <= 1e-10, e
    again = mbl.entanglement_entropy(chain, l_a, torch.from_numpy(V.copy()).to(DEV)).cpu().numpy()
    assert np.array_equal(S, again)


def test_not_finite_and_many_columns(mbl):
    L = 8
    st = ham.basis(L, 4)
    rng = np.random.default_rng(3)
    V = rng.normal(size=(st.size, 9000))  # 45,000 (vector, p) pairs: two launches
    V[3, 7] = np.nan
    V[5, 8] = np.inf
    chain = mbl.make_chain(L, np.zeros(L))
    S = mbl.entanglement_entropy(chain, 4, torch.from_numpy(V).to(DEV)).cpu().numpy()
    assert math.isnan(S[7]) and math.isnan(S[8])
    for e in (0, 6, 9, 4500, 8999):
        assert abs(S[e] - obs.entanglement_entropy(st, V[:, e], 4)) <= 1e-10


# cuts of small Grams and long sums, one kernel and its combine (2 launches), beside the five kernels
@pytest.mark.parametrize("L,n_up,l_a,launches", [
    (8, 4, 2, 2), (10, 5, 3, 2), (14, 7, 3, 2), (16, 8, 4, 2), (18, 9, 4, 2), (20, 10, 5, 2), (20, 10, 16, 2), (12, 1, 6, 2), (20, 7, 6, 2), (10, 5, 4, 2),
    (10, 5, 5, 5), (12, 6, 5, 5), (14, 7, 7, 5), (18, 9, 7, 5)])
def test_small_grams(mbl, L, n_up, l_a, launches):
    rng = np.random.default_rng(L * 17 + l_a)
    st = ham.basis(L, n_up)
    V = _columns(L, st, rng)
    V = np.concatenate([V, np.zeros((st.size, 2))], axis=1)
    V[st.size // 2, 5] = np.nan
    chain = mbl.make_chain(L, np.zeros(L), 1.0, False, n_up)
    before = mbl.binding.kernel_launch_count()
    S = mbl.entanglement_entropy(chain, l_a, torch.from_numpy(V.copy()).to(DEV)).cpu().numpy()
    assert mbl.binding.kernel_launch_count() - before == launches
    for e in range(4):
        assert abs(S[e] - obs.entanglement_entropy(st, V[:, e], l_a)) <= 1e-10, e
    assert math.isnan(S[4]) and math.isnan(S[5])  # a zero column, a NaN
