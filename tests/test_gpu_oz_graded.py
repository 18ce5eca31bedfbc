"""Larger ends of complex128 bonds whose contraction index is graded: near the canonical form
Gamma[r][k] grows like 1 / lambda_k in rows of small lambda on the other legs, and the factor it
meets in the update shrinks like lambda_k.  The updated tensor has to hold the digits that FP64
multiply-adds give it, at the first D of every operand layout of the tensor-core passes.
"""
import numpy as np
import pytest
import torch

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps
# site 0 joins three legs; its bond to site 1 (one more leg) is the only edge of class 0
GRAPH = (5, np.array([[0, 1], [0, 2], [0, 3], [1, 4]], dtype=np.int32))


def _random(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


def _kick(t, th):
    c, s = np.cos(th / 2), np.sin(th / 2)
    return np.stack([c * t[0] - 1j * s * t[1], c * t[1] - 1j * s * t[0]])


def _handle(D, gammas, lams):
    g = gpu_lib()([GRAPH], D, dtype="c128")
    g.reset()
    for i, t in gammas.items():
        g.site_tensor(0, i)[0].copy_(torch.from_numpy(t))
    for e, v in lams.items():
        g.lambda_tensor(0, e).copy_(torch.from_numpy(v))
    torch.cuda.synchronize()
    return g


@pytest.mark.parametrize("lam_min", [1e-3, 1e-6, 1e-10])
@pytest.mark.parametrize("D", [17, 32, 33, 64, 65, 128])
def test_graded_tensor_keeps_its_digits(D, lam_min):
    """Gamma_a'[r, k'] = sum_x Psi[r, x] V[x, k'] / s_k', with Psi the gated two-site tensor (rows of
    end a not weighted) and V read back from the updated end b (Gamma_b' = conj(V) / lambda_other),
    so no gauge is left open and no accuracy of the SVD enters.  The library's path through
    Y = lambda F conj(V) / s sums 2D and then D products, the reference D and then 2D, so both stay
    within (2D + D + 16) eps of sum_k |A~[r, k]| lambda_k |F_k| / s_k', 9e-14 at D = 128; s_0 from a
    LAPACK SVD scales the normalised lambda (1e-13).  Held to 1e-12."""
    rng = np.random.default_rng(D)
    lam = np.exp(np.log(lam_min) * np.arange(D) / (D - 1))
    lam4 = np.linspace(1.0, 0.5, D)
    cap = np.minimum(1 / np.maximum(lam[:, None, None] * lam[None, :, None], 1e-300),
                     1 / np.maximum(lam[:, None, None] * lam[None, None, :], 1e-300))
    cap = np.minimum(cap, 1 / (lam[None, :, None] * lam[None, None, :]))  # [k][r2][r3]
    g0 = _random(rng, 2, D, D, D) * cap / D
    g1 = _random(rng, 2, D, D) / np.sqrt(D)
    g = _handle(D, {0: g0, 1: g1}, {0: lam, 1: lam, 2: lam, 3: lam4})
    th = 0.7
    g.kick(torch.tensor([th], dtype=torch.float64, device="cuda"))
    g.zz_layer(0)
    assert g.status() == 0
    A1 = g.site_tensor(0, 0)[0].cpu().numpy().transpose(0, 2, 3, 1).reshape(2, D * D, D)
    B1 = g.site_tensor(0, 1)[0].cpu().numpy()  # [t][k'][x]
    new = g.lambda_tensor(0, 0).cpu().numpy()
    g.close()
    A = _kick(g0, th).transpose(0, 2, 3, 1).reshape(2, D * D, D)
    F = _kick(g1, th) * lam4  # [t][k][x]
    w = (lam[:, None] * lam[None, :]).reshape(-1)
    phase = np.exp(1j * np.pi / 4 * np.array([[1, -1], [-1, 1]]))
    psi = np.einsum("st,srk,tkx->srtx", phase, A * lam, F, optimize=True).reshape(2, D * D, 2 * D)
    s0 = np.linalg.svd((psi * w[None, :, None]).reshape(-1, 2 * D), compute_uv=False)[0]
    s = new / new.max() * s0
    on = s > 0
    V = (np.conj(B1) * lam4).transpose(0, 2, 1).reshape(2 * D, D)  # V[(t, x)][k']
    ref = psi @ V[:, on] / s[on]
    scale = (np.abs(A) * (lam * np.sqrt((np.abs(F) ** 2).sum((0, 2))))).sum(2)  # [s][r]
    err = np.abs(A1[:, :, on] - ref) * s[on] / scale[:, :, None]
    assert err.max() <= 1e-12


@pytest.mark.parametrize("D", [17, 33, 65])
def test_failed_bond_leaves_the_larger_end_unrounded(D):
    """A bond whose core is not finite keeps its tensors; only the pending kick of the larger end is
    applied, two multiply-adds an element whatever the rest of its row holds."""
    rng = np.random.default_rng(D)
    g0 = _random(rng, 2, D, D, D) * 10.0 ** rng.uniform(-30, 0, (2, D, D, D))
    g1 = _random(rng, 2, D, D)
    g1[0, 1, 2] = np.nan
    lam = np.linspace(1.0, 0.5, D)
    lam0 = np.where(np.arange(D) < D // 2, lam, 0.0)
    for th in (0.0, 0.7):
        g = _handle(D, {0: g0, 1: g1}, {0: lam0, 1: lam, 2: lam, 3: lam})
        g.kick(torch.tensor([th], dtype=torch.float64, device="cuda"))
        g.zz_layer(0)
        assert g.status() == 2
        got, ref = g.site_tensor(0, 0)[0].cpu().numpy(), _kick(g0, th)
        assert np.array_equal(g.lambda_tensor(0, 0).cpu().numpy(), lam0)
        g.close()
        part = np.abs(g0) + np.abs(g0[::-1])  # an element's two terms
        assert (np.abs(got - ref) <= 4 * EPS * part).all()
        assert th or np.array_equal(got, g0)
