"""The FP32 warm start of the complex128 bond SVD and what makes its basis good to FP64, at the
edges of their tilings: columns of 8, 16 and 32 lanes (lengths 2D to 64, 128 and 256), D = 23 | 24
where the products of the core go from FP64 multiply-adds to digit products on the tensor
cores and the simultaneous correction begins, rank-deficient and pairwise degenerate spectra,
and a warm start that ends at its sweep cap.  One Trotter step of a random state against the oracle,
tolerance 1e-10 on <Z> as for the complex128 path elsewhere (mixed: 1e-4).
"""
import numpy as np
import pytest
import torch

from oracle import su
from workloads import heavy_hex

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


def _step(D, dtype="c128", spectrum=None, settings=None):
    # beyond D = 17 three arms of two bonds: the inner ones have a core of 2D columns
    arms = (7, np.array([[0, 1], [0, 2], [0, 3], [1, 4], [2, 5], [3, 6]], dtype=np.int32))
    n, edges = heavy_hex(3, 7) if D <= 17 else arms
    p = su.GPEPS(n, edges, D)
    rng = np.random.default_rng(D)
    for i in range(p.n):
        shape = p.gamma[i].shape
        p.gamma[i] = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / 2
        if dtype == "mixed":
            p.gamma[i] = p.gamma[i].astype(np.complex64).astype(np.complex128)
    lam = np.exp(-rng.uniform(0.7, 1.05, (len(p.edges), 1)) * np.sqrt(np.arange(D)))
    if spectrum:
        spectrum(lam)
    p.lam = lam / np.linalg.norm(lam, axis=1, keepdims=True)
    g = gpu_lib()([(n, edges)], D, dtype=dtype)
    if settings:
        settings(g)
    for i in range(n):
        t = g.site_tensor(0, i)[0]
        t.copy_(torch.from_numpy(p.gamma[i]).to(t.dtype))
    for e in range(len(p.edges)):
        g.lambda_tensor(0, e).copy_(torch.from_numpy(p.lam[e]))
    torch.cuda.synchronize()
    g.step(1, torch.tensor([0.7], dtype=torch.float64, device="cuda"))
    z = g.expect_z()[0].cpu().numpy()
    assert g.status() == 0
    g.close()
    p.step(0.7)
    return np.abs(z - p.expect_z()).max()


@pytest.mark.parametrize("cap", [0, 2])
@pytest.mark.parametrize("dtype,tol", [("mixed", 1e-4), ("c128", 1e-10)])
def test_a_capped_warm_start_leaves_the_work_to_the_fp64_sweeps(dtype, tol, cap):
    assert _step(16, dtype, settings=lambda g: g.set_jacobi(max_sweeps32=cap)) <= tol


@pytest.mark.parametrize("tol32", [1e-9, 1e-2])
def test_a_warm_start_tolerance_out_of_range_is_brought_into_it(tol32):
    assert _step(16, settings=lambda g: g.set_jacobi(tol32=tol32)) <= 1e-10


@pytest.mark.parametrize("D", [3, 4, 9, 23, 24, 31, 32, 33, 64, 65])
def test_step_of_a_random_state(D):
    assert _step(D) <= 1e-10


def _rank5(lam):
    lam[:, 5:] = 0.0


def _pairs(lam):
    lam[:, 1::2] = lam[:, 0:-1:2]


@pytest.mark.parametrize("D", [24, 32, 64])
@pytest.mark.parametrize("spectrum", [_rank5, _pairs])
def test_step_of_a_degenerate_state(D, spectrum):
    assert _step(D, spectrum=spectrum) <= 1e-10
