"""Steps of the complex128 bond SVD on their own (gpeps_selftest_core)."""
import ctypes
import math

import numpy as np
import pytest
import torch

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


def _run(which, a, b):
    gpu_lib()
    from paper_2309_15642_gb300 import _abi
    x, y = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, b))
    out = torch.empty_like(x)
    assert _abi.load().gpeps_selftest_core(which, len(a), x.data_ptr(), y.data_ptr(), out.data_ptr(),
                                           ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _two_products(x, y):
    """x y as a sum of two doubles (Dekker, with Veltkamp's splitting)."""
    def split(v):
        t = 134217729.0 * v
        hi = t - (t - v)
        return hi, v - hi
    p, (xh, xl), (yh, yl) = x * y, split(x), split(y)
    return p, ((xh * yh - p) + xh * yl + xl * yh) + xl * yl


@pytest.mark.parametrize("n", [48, 64, 128, 256])
def test_digit_product_is_no_less_accurate_than_fp64(n):
    """Gaussian rows: every real output against its exact value, in units of 2^-53 of the two rows'
    powers of two.  They have to be no worse than FP64 products summed in order, and unbiased
    within five standard errors."""
    rng = np.random.default_rng(n)
    a, b = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n)) for _ in range(2))
    got = _run(0, a, b)
    rows = rng.permutation(n)[:16]
    unit = [2.0 ** np.frexp(np.maximum(np.abs(v.real), np.abs(v.imag)).max(1))[1] for v in (a, b)]
    err, plain = [], []
    for i in rows:
        # re: (ar, ai) . (br, bi), im: (ar, -ai) . (bi, br)
        for part, x, y in ((got[i].real, np.r_[a[i].real, a[i].imag], np.c_[b.real, b.imag]),
                           (got[i].imag, np.r_[a[i].real, -a[i].imag], np.c_[b.imag, b.real])):
            p, q = _two_products(x[None, :], y)
            scale = unit[0][i] * unit[1] * 2.0 ** -53
            exact = [math.fsum(np.r_[u, v]) for u, v in zip(p, q)]
            rest = [math.fsum(np.r_[u, v, -w]) for u, v, w in zip(p, q, exact)]
            err.append(((part - exact) - rest) / scale)
            s = np.zeros(n)
            for k in range(x.size):
                s = s + p[:, k]
            plain.append(((s - exact) - rest) / scale)
    err, plain = np.array(err), np.array(plain)
    rms, ref = np.sqrt((err ** 2).mean()), np.sqrt((plain ** 2).mean())
    assert rms <= ref
    assert abs(err.mean()) <= 5 * rms / np.sqrt(err.size)


def test_rejects_bad_arguments():
    gpu_lib()
    from paper_2309_15642_gb300 import _abi
    lib = _abi.load()
    x = torch.zeros(64, dtype=torch.float64, device="cuda").data_ptr()
    for which, n, p in ((7, 4, x), (0, 3, x), (0, 0, x), (0, 258, x), (0, 4, None)):
        assert lib.gpeps_selftest_core(which, n, p, p, p, None) == _abi.GPEPS_EINVAL
