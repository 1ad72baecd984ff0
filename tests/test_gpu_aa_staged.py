"""The in-place step's persistent TMA-staged form (FP32 domains whose buffer
exceeds L2) against the same step pulling its populations: bit for bit, over both
parities, ragged last tiles and the tiles on the periodic edge.
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


def _state(HLBM, c, steps):
    g = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params)
    if c.gfield is not None:
        g.set_force_field(c.gfield[:, :, 0], "profile")
    g.init(c.rho, c.u, c.theta)
    for n in steps:
        g.step(n)
    s = g.save()
    g.close()
    return np.frombuffer(s, np.uint8)


@pytest.mark.parametrize("kind", ["kolmogorov", "thermal", "droplet"])
@pytest.mark.parametrize("nx,ny", [(1024, 640), (900, 901), (44, 14800)])
def test_staged_in_place_step_equals_pulled(HLBM, monkeypatch, kind, nx, ny):
    if kind == "kolmogorov":
        c = W.kolmogorov(nx=nx, ny=ny, g0=1e-4)
    elif kind == "thermal":
        c = W.thermal_decay(nx=nx, ny=ny, tau_hat=0.7, Pr=0.71)
    else:
        c = W.droplet(nx=nx, ny=ny, r0=0.3 * min(nx, ny), Tr=0.9, k=1.5672)
    c.params = dict(c.params, lag=True)
    steps = (1, 2, 36)      # single launches of both parities, then a graph
    a = _state(HLBM, c, steps)
    monkeypatch.setenv("HLBM_NO_TMA", "1")
    b = _state(HLBM, c, steps)
    assert np.array_equal(a, b)
