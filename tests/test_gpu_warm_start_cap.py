"""A complex128 warm start that ends at its sweep cap hands on what it has: one Trotter step of a
random state, the FP64 sweeps counted.  Thrown away, five FP32 sweeps leave the FP64 ones a whole
solve (11, 15 and 21 sweeps a bond); an accumulated rotation product, kept, left 6.1, 9.0 and 13.6 of
the same states.
"""
import numpy as np
import pytest
import torch

from workloads import heavy_hex

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


def _steps(D, caps):
    n, edges = heavy_hex(3, 7)
    rng = np.random.default_rng(D)
    g = gpu_lib()([(n, edges)], D, dtype="c128")
    for i in range(n):
        t = g.site_tensor(0, i)[0]
        t.copy_(torch.from_numpy((rng.standard_normal(t.shape) + 1j * rng.standard_normal(t.shape)) / 2))
    for e in range(len(edges)):
        lam = np.exp(-rng.uniform(0.7, 1.05) * np.sqrt(np.arange(D)))
        g.lambda_tensor(0, e).copy_(torch.from_numpy(lam / np.linalg.norm(lam)))
    torch.cuda.synchronize()
    saved, out = g.state.clone(), {}
    for cap in caps:
        g.set_jacobi(max_sweeps32=cap)
        g.reset()
        g.load_state(saved)
        g.step(1, torch.tensor([0.7], dtype=torch.float64, device="cuda"))
        z = g.expect_z()[0].cpu().numpy()
        assert g.status() == 0
        out[cap] = z, g.sweeps()[0] / g.sweeps()[2]
    g.close()
    return out


@pytest.mark.parametrize("D,most", [(16, 6.1), (32, 9.0), (64, 13.6)])
def test_capped_warm_start_shortens_the_fp64_sweeps(D, most):
    out = _steps(D, (5, 20))
    assert out[5][1] <= most
    assert np.abs(out[5][0] - out[20][0]).max() <= 1e-10
