"""A schedule changed between calls (hlbm_set_tile after steps have run): the next
call of any kind gives what a context with that schedule from the start gives.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def HLBM():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_10751_gb300 as pkg
    pkg.build()
    from paper_2411_10751_gb300.solver import HLBM as cls
    return cls


def _context(HLBM, c, schedule):
    g = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params)
    g.set_tile(*schedule)
    if c.gfield is not None:
        g.set_force_field(c.gfield, "field")
    g.init(c.rho, c.u, c.theta)
    return g


@pytest.mark.parametrize("K", [1, 4])
def test_adjoint_after_a_change_of_schedule(HLBM, K):
    c = W.kolmogorov(nx=224, ny=200, g0=1e-4)
    ref = _context(HLBM, c, (8, 2, 2))
    ref.step(2)
    loss0, grad0 = ref.adjoint(10, K)
    g = _context(HLBM, c, (16, 2, 2))     # 91 tiles and as many CTAs per launch; then 175
    g.step(2)                             # 2 x 182 values of the counter: 14 into the period of 350
    g.set_tile(8, 2, 2)
    loss, grad = g.adjoint(10, K)
    assert loss == loss0
    assert np.array_equal(grad.cpu().numpy(), grad0.cpu().numpy())
    assert g.save() == ref.save()
    ref.close()
    g.close()


@pytest.mark.parametrize("first,then", [((16, 2, 3), (8, 2, 3)), ((8, 2, 3), (4, 1, 3)), ((8, 1, 3), (16, 1, 3))])
def test_multi_step_kernel_after_a_change_of_rows(HLBM, first, then):
    """Against the same steps on the same tiles by the kernel of one launch per step
    (other tiles round theta on their frames differently)."""
    c = W.thermal_decay(nx=128, ny=96)
    ref = _context(HLBM, c, first[:2] + (2,))
    ref.step(7)
    ref.set_tile(*then[:2], 2)
    ref.step(10)
    g = _context(HLBM, c, first)
    g.step(7)
    g.set_tile(*then)
    g.step(10)
    g.synchronize()
    assert g.save() == ref.save()
    ref.close()
    g.close()
