"""Complex128 Gram and update passes on the tensor cores (integer digit products): one Trotter
step of a random full-rank state at the edges of the tilings (D = 16 the smallest, 32 | 33 and
64 | 65 where the operand layout changes, odd and ragged sizes, 128 the largest) against the
oracle, every qubit and every lambda.  Tolerances as for the complex128 path elsewhere: 1e-10
on <Z>, 1e-9 on lambda.
"""
import numpy as np
import pytest
import torch

from oracle import su
from workloads import heavy_hex

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


def _random_state(p, rng):
    for i in range(p.n):
        shape = p.gamma[i].shape
        p.gamma[i] = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / 2
    lam = np.exp(-rng.uniform(0.7, 1.05, (len(p.edges), 1)) * np.sqrt(np.arange(p.D)))
    p.lam = lam / np.linalg.norm(lam, axis=1, keepdims=True)


def _load(g, p):
    for i in range(p.n):
        g.site_tensor(0, i)[0].copy_(torch.from_numpy(p.gamma[i]))
    for e in range(len(p.edges)):
        g.lambda_tensor(0, e).copy_(torch.from_numpy(p.lam[e]))
    torch.cuda.synchronize()


@pytest.mark.parametrize("D", [16, 17, 31, 32, 33, 64, 65, 128])
def test_step_of_a_random_state_matches_oracle(D):
    # the arms of one degree-3 site (bond leg first, middle and last in its tensor) and their
    # degree-2 and degree-1 neighbours; beyond D = 33 the smallest such graph
    n, edges = heavy_hex(3, 7) if D <= 33 else (4, np.array([[0, 1], [1, 2], [1, 3]], dtype=np.int32))
    p = su.GPEPS(n, edges, D)
    _random_state(p, np.random.default_rng(D))
    g = gpu_lib()([(n, edges)], D, dtype="c128")
    _load(g, p)
    g.step(1, torch.tensor([0.7], dtype=torch.float64, device="cuda"))
    z = g.expect_z()[0].cpu().numpy()
    assert g.status() == 0
    p.step(0.7)
    assert np.abs(z - p.expect_z()).max() <= 1e-10
    lam = np.stack([g.lambdas(0, e) for e in range(len(edges))])
    assert np.abs(lam - p.lambdas()).max() <= 1e-9
    g.close()


def test_non_finite_input_is_reported():
    """A NaN in a site tensor still raises GPEPS_FLAG_NUMERIC on the bonds that read it (the digits
    of a NaN are integers: its row's exponent marks it)."""
    n, edges = heavy_hex(3, 7)
    p = su.GPEPS(n, edges, 16)
    _random_state(p, np.random.default_rng(1))
    g = gpu_lib()([(n, edges)], 16, dtype="c128")
    i = next(v for v in range(n) if len(p.nb[v]) == 3)
    p.gamma[i].flat[5] = np.nan
    _load(g, p)
    g.step(1, torch.tensor([0.7], dtype=torch.float64, device="cuda"))
    assert g.status() & 2
    g.close()
