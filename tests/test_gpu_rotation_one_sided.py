"""What the FP64 sweeps of the complex128 bond SVD use of a rotation (gpeps_selftest_rotation, which
3): tau = t / |g|, c, u = 1 + t^2 and w = t |g|, by which the squared norms of the pair change,
against the textbook formulas in CUDA's FP64 functions.  tau comes from FP32 and one Newton step
(relative error about 1e-7 x 1e-7: held to 5e-13), c from u by a third-order step (a few roundings:
c^2 u = 1 to 4 eps), w is a rounded product of tau.
"""
import numpy as np
import pytest

from .test_gpu_rotation import EPS, _inputs, _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(-12, 0), (-120, -100), (100, 120), (-150, 150)])
def test_one_sided_rotation_results(lo, hi):
    x = _inputs(np.random.default_rng(5), 4096, lo, hi, False)
    x = x[np.abs(np.log10(np.hypot(x[:, 2], x[:, 3]))) < 150]
    tau, c, u, w, tr, cr, ur, wr = _run(3, x).T
    assert (np.abs(tau - tr) <= 5e-13 * np.abs(tr)).all()
    assert np.abs(c * c * u - 1).max() <= 4 * EPS
    assert (np.abs(u - ur) <= 1e-12 * ur).all()
    assert (np.abs(c - cr) <= 5e-13 * cr).all()
    g2 = x[:, 2] ** 2 + x[:, 3] ** 2
    assert (np.abs(w - g2 * tau) <= 4 * EPS * np.abs(w)).all()
    # the norms after the rotation: no larger sum, and the determinant a b - |g|^2 within rounding
    # of its terms and the angle's error
    a, b = x[:, 0], x[:, 1]
    m = np.maximum(a, b)
    det = ((a - w) / m) * ((b + w) / m)
    assert (np.abs(det - (a * (b / m) - g2 / m) / m) <= 2e-12).all()


@pytest.mark.parametrize("a,b", [(1.5e308, 1.0), (1.0, 1.5e308), (9e307, 1e300), (1.7e308, 1.7e308), (3e307, 1e-300)])
def test_one_sided_rotation_at_the_end_of_the_range(a, b):
    """Squared norms up to the largest double: t underflows or is that of equal norms; nothing wraps."""
    g = 1e150
    tau, c, u, w, tr, cr, ur, wr = _run(3, np.array([[a, b, g, 0.0], [a, b, 0.0, -g]])).T
    assert (np.abs(tau - tr) <= 5e-13 * np.abs(tr) + 2.3e-308).all()
    assert (np.abs(c - cr) <= 5e-13).all() and (np.abs(u - ur) <= 1e-12 * ur).all()
    assert (np.abs(w - wr) <= 4 * EPS * max(a, b) + 5e-13 * np.abs(wr)).all()
