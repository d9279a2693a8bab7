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
