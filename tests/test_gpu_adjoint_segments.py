"""hlbm_adjoint_run over checkpoint intervals whose segments end in every way (a last
segment of one step, one segment, as many as steps, odd and even step counts): the loss
and gradient of the run that keeps every state, and the context left at step T.
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


def _case(which):
    rng = np.random.default_rng(8)
    if which == "d2q37":
        c = W.kolmogorov(nx=52, ny=37)
        c.gfield = W.fp32(2e-4 * (2 * rng.random((2, 37, 52)) - 1))
        return c
    n = {"d3q39_gather": 21, "d3q39_rows": 32}[which]
    c = W.taylor_green_3d(n=32, tau_hat=0.6, Ma=0.1)
    sl = (slice(0, 9), slice(0, 11), slice(0, n))
    c.rho, c.theta = c.rho[sl].copy(), c.theta[sl].copy()
    c.u = c.u[(slice(None),) + sl].copy()
    c.nz, c.ny, c.nx = c.rho.shape
    c.gfield = W.fp32(2e-4 * (2 * rng.random((3,) + c.rho.shape) - 1))
    return c


def _context(HLBM, c):
    g = HLBM(c.lattice, c.nx, c.ny, c.nz, c.tau_hat, c.params)
    g.set_force_field(c.gfield, "field")
    g.init(c.rho, c.u, c.theta)
    return g


@pytest.mark.parametrize("which", ["d2q37", "d3q39_gather", "d3q39_rows"])
@pytest.mark.parametrize("T,K", [(1, 2), (2, 2), (3, 2), (4, 2), (7, 2), (8, 2), (7, 3), (9, 4), (6, 5), (6, 6), (5, 9)])
def test_segments_do_not_change_gradient_or_final_state(HLBM, which, T, K):
    c = _case(which)
    g = _context(HLBM, c)
    g.step(3)                      # the run starts from the other buffer
    g0 = _context(HLBM, c)
    g0.step(3)
    loss, grad = g.adjoint(T, K)
    loss0, grad0 = g0.adjoint(T, 1)
    assert loss == loss0
    assert np.array_equal(grad.cpu().numpy(), grad0.cpu().numpy())
    f = _context(HLBM, c)
    f.step(3)
    f.step(T)
    assert g.step_count == f.step_count == g0.step_count
    assert g.save() == f.save() == g0.save()
    for s in (g, f):               # and both go on alike
        s.step(2)
    assert g.save() == f.save()
    for s in (g, g0, f):
        s.close()
