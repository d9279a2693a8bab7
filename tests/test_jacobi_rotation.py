"""The FP64 Jacobi rotation of the small eigensolver, restated in numpy: t from FP32, then
c = 1 / sqrt(1 + t^2) by two FP64 Newton steps from an FP32 start.  It has to be orthogonal to
FP64 and to leave a small fraction of a_pq, whatever the sizes of the three entries."""
import numpy as np
import pytest


def _rotation(apq, app, aqq):
    d = aqq - app
    e = np.maximum(np.frexp(d)[1], np.frexp(apq)[1])
    tau = np.float32(np.ldexp(d, -e)) / (np.float32(2) * np.float32(np.ldexp(apq, -e)))
    t = np.copysign(np.float32(1), tau) / (np.abs(tau) + np.sqrt(tau * tau + np.float32(1)))
    t = t.astype(np.float64)
    u = t * t + 1.0
    y = (np.float32(1) / np.sqrt(u.astype(np.float32))).astype(np.float64)
    y *= 1.0 + 2e-7  # the hardware's reciprocal root: within 2 ulp
    for _ in range(2):
        y = y * (1.5 - 0.5 * u * (y * y))
    return y, t * y


@pytest.mark.parametrize("spread", [0, 3, 12, 28])
def test_rotation_is_orthogonal_and_annihilates(spread):
    rng = np.random.default_rng(spread)
    size = lambda: rng.normal(size=20000) * 2.0 ** rng.uniform(-spread, spread, 20000)  # noqa: E731
    apq, app, aqq = size(), size(), size()
    c, s = _rotation(apq, app, aqq)
    assert np.abs(c * c + s * s - 1.0).max() <= 4 * np.finfo(np.float64).eps
    left = (c * c - s * s) * apq + c * s * (app - aqq)
    # t is right to a few FP32 roundings: a_pq's share and the rotated diagonal's
    assert np.all(np.abs(left) <= 1e-6 * np.abs(apq) + 4e-16 * (np.abs(app) + np.abs(aqq)))


def _guarded(apq, app, aqq):
    """The rotation with its choice: beyond a difference of 2^60 times a_pq the FP64 formula."""
    d = aqq - app
    wide = np.frexp(d)[1] - np.frexp(apq)[1] > 60
    with np.errstate(over="ignore", invalid="ignore", divide="ignore"):
        c, s = _rotation(apq, app, aqq)
    tau = d / (2.0 * apq)
    t = np.copysign(1.0, tau) / (np.abs(tau) + np.sqrt(1.0 + tau * tau))
    ce = 1.0 / np.sqrt(1.0 + t * t)
    return np.where(wide, ce, c), np.where(wide, t * ce, s)


@pytest.mark.parametrize("log_tau", [50, 58, 59, 60, 61, 62, 63, 64, 65, 70, 90, 99, 100, 101, 110])
def test_rotation_of_a_graded_pair(log_tau):
    rng = np.random.default_rng(log_tau)
    apq = rng.normal(size=5000)
    apq[np.abs(apq) < 1e-3] = 1.0
    app, aqq = np.zeros(5000), rng.uniform(1.0, 4.0, 5000) * 2.0 ** log_tau
    c, s = _guarded(apq, app, aqq)
    assert np.all(s != 0.0)
    # a_pq is annihilated: t = a_pq / a_qq there, to a few FP32 roundings
    left = (c * c - s * s) * apq + c * s * (app - aqq)
    assert np.all(np.abs(left) <= 1e-6 * np.abs(apq))
