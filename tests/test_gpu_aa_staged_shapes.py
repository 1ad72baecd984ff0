"""The in-place step's staged form against the pulled one, bit for bit, on shapes that
its rule takes it for: just above its sizes, ragged last tiles in both directions,
narrow domains of whole tile columns where no tile is boxed.
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


@pytest.mark.parametrize("kind", ["kolmogorov", "thermal", "droplet"])
@pytest.mark.parametrize("nx,ny", [(1024, 716), (900, 813), (200, 3701), (32, 22900), (96, 7700), (22908, 32)])
def test_staged_in_place_step_equals_pulled(HLBM, monkeypatch, kind, nx, ny):
    assert 37 * nx * ny * 4 >= 108e6
    if kind == "kolmogorov":
        c = W.kolmogorov(nx=nx, ny=ny, g0=1e-4)
    elif kind == "thermal":
        c = W.thermal_decay(nx=nx, ny=ny, tau_hat=0.7, Pr=0.71)
    else:
        c = W.droplet(nx=nx, ny=ny, r0=0.3 * min(nx, ny), Tr=0.9, k=1.5672)
    c.params = dict(c.params, lag=True)

    def state():
        g = HLBM(c.lattice, nx, ny, 1, c.tau_hat, c.params)
        if c.gfield is not None:
            g.set_force_field(c.gfield[:, :, 0], "profile")
        g.init(c.rho, c.u, c.theta)
        for n in (1, 2, 33):       # single launches of both parities, then a graph
            g.step(n)
        s = g.save()
        g.close()
        return np.frombuffer(s, np.uint8)

    a = state()
    monkeypatch.setenv("HLBM_NO_TMA", "1")
    assert np.array_equal(a, state())
