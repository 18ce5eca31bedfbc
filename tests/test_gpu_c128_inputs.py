"""Complex128 at the sizes where its code paths part: values that are not finite through the digit
passes (their operand layouts begin at D = 17, 33 and 65), and the fused step, which complex128 runs
up to D = 16, against the layered launches bit for bit.
"""
import numpy as np
import pytest
import torch

from workloads import EAGLE, heavy_hex

from ._gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("D", [17, 33, 65])
def test_non_finite_input_is_reported(D, value):
    """Digits are integers: only its row's exponent marks a value that is not finite.  Class 0 holds
    the bond of sites 0 and 1 alone; it is reported and keeps lambda and its tensors but for the two
    elements that the kick (of angle zero: a product with 0) mixes with the value; the next class
    fails as well (site 0 still holds it)."""
    n, edges = 5, np.array([[0, 1], [0, 2], [0, 3], [1, 4]])
    rng = np.random.default_rng(D)
    g = gpu_lib()([(n, edges)], D, dtype="c128")
    g.reset()
    for v in range(n):
        t = g.site_tensor(0, v)[0]
        t.copy_(torch.from_numpy(rng.standard_normal(t.shape) + 1j * rng.standard_normal(t.shape)))
    for e in range(len(edges)):
        g.lambda_tensor(0, e).copy_(torch.from_numpy(np.linspace(1.0, 0.5, D)))
    g.site_tensor(0, 0)[0][1, D - 1, 0, D // 2] = complex(0.0, value)
    torch.cuda.synchronize()
    before = g.state.clone()
    for c in range(2):
        g.zz_layer(c)
        assert g.status() == 2
        if c == 0:
            after = g.state.clone()
            for state in (before, after):
                g.state.copy_(state)
                g.site_tensor(0, 0)[0][:, D - 1, 0, D // 2] = 0
                state.copy_(g.state)
            assert torch.equal(after, before)
            g.site_tensor(0, 0)[0][1, D - 1, 0, D // 2] = complex(0.0, value)
            torch.cuda.synchronize()
    g.close()


def test_finite_neighbours_of_a_failed_bond_are_updated():
    """The value stays where it was: a bond that does not touch its site is updated as without it."""
    n, edges = heavy_hex(3, 7)
    D, rng = 17, np.random.default_rng(3)
    tensors = {}
    states = []
    for bad in (False, True):
        g = gpu_lib()([(n, edges)], D, dtype="c128")
        g.reset()
        for v in range(n):
            t = g.site_tensor(0, v)[0]
            if v not in tensors:
                tensors[v] = torch.from_numpy(rng.standard_normal(t.shape) + 1j * rng.standard_normal(t.shape))
            t.copy_(tensors[v])
        for e in range(len(edges)):
            g.lambda_tensor(0, e).copy_(torch.from_numpy(np.linspace(1.0, 0.5, D)))
        if bad:
            g.site_tensor(0, 0)[0].view(-1)[3] = complex(np.inf, 0.0)
        torch.cuda.synchronize()
        g.zz_layer(0)
        assert g.status() == (2 if bad else 0)
        states.append([g.site_tensor(0, v)[0].clone() for v in range(n)])
        near = {0} | set(g.site_tensor(0, 0)[1])
        g.close()
    for v in range(n):
        if v not in near:
            assert torch.equal(states[0][v], states[1][v])


@pytest.mark.parametrize("D,schedule", [(4, 4), (9, 4), (16, 4), (4, 5), (16, 5)])
def test_complex128_fused_step_bit_identical(D, schedule):
    n, edges = heavy_hex(*EAGLE)
    states = []
    for s in (0, schedule):
        g = gpu_lib()([(n, edges)], D, dtype="c128")
        g.set_schedule(s)
        g.reset()
        m = g.step(7, torch.tensor([0.7], dtype=torch.float64, device="cuda"))
        assert g.status() == 0
        assert (g.pass_cycles()[0] > 0) == (s > 0)  # the Gram pass ran inside the fused step, or did not
        states.append((m.clone(), g.state.clone()))
        g.close()
    assert torch.equal(states[0][0], states[1][0]) and torch.equal(states[0][1], states[1][1])


@pytest.mark.parametrize("schedule", [1, 2, 3, 4, 5])
def test_complex128_schedules_bit_identical(schedule):
    """D = 33 and 64 on every schedule that the handle takes, classes larger than the SM count."""
    n, edges = heavy_hex(*EAGLE)
    for D, copies in ((33, 9), (64, 4)):
        states = []
        for s in (0, schedule):
            g = gpu_lib()([(n, edges)] * copies, D, dtype="c128")
            try:
                g.set_schedule(s)
            except RuntimeError:
                assert s == 5  # three CTAs of the fused step do not fit
                g.close()
                return
            g.reset()
            m = g.step(5, torch.full((copies,), 0.7, dtype=torch.float64, device="cuda"))
            assert g.status() == 0
            states.append((m.clone(), g.state.clone()))
            g.close()
        assert torch.equal(states[0][0], states[1][0]) and torch.equal(states[0][1], states[1][1])
