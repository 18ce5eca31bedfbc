"""A complex128 colour class that runs in groups of bonds because state and scratch would pass 240 GiB
(3 x 1121 qubits at D = 128: groups of at most 304 bonds): instances that hold the same tensors
end bit for bit alike, whichever group their bonds fell into.
"""
import pytest
import torch

from workloads import CONDOR, heavy_hex

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


def test_groups_of_a_class_give_the_same_bits():
    GPEPS = gpu_lib()
    if torch.cuda.mem_get_info()[0] < 160e9:
        pytest.skip("needs 150 GB")
    (n, edges), D = heavy_hex(*CONDOR), 128
    copies = 3
    g = GPEPS([(n, edges)] * copies, D, dtype="c128")
    gen = torch.Generator(device="cuda").manual_seed(5)
    for v in range(n):
        t = g.site_tensor(0, v)[0]
        t.copy_(torch.randn(t.shape, generator=gen, device="cuda", dtype=t.dtype))
        for k in range(1, copies):
            g.site_tensor(k, v)[0].copy_(t)
    for e in range(len(edges)):
        lam = torch.rand(D, generator=gen, device="cuda", dtype=torch.float64)
        for k in range(copies):
            g.lambda_tensor(k, e).copy_(lam)
    torch.cuda.synchronize()
    before = g.lambda_tensor(0, 0).clone()
    ms = g.zz_layer_profiled(0)
    assert g.status() == 0
    assert g.sweeps()[2] > 3 * 304 and min(ms) > 0
    for k in range(1, copies):
        for v in range(n):
            assert torch.equal(g.site_tensor(0, v)[0], g.site_tensor(k, v)[0])
        for e in range(len(edges)):
            assert torch.equal(g.lambda_tensor(0, e), g.lambda_tensor(k, e))
    assert not torch.equal(before, g.lambda_tensor(0, 0))
    g.close()
