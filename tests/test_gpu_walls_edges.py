"""Wall-bounded step at the edges of its launches: domains of the fewest rows and
columns, block rows and columns that are cut short, both wall kinds, with and
without the thermal source; and a split run (the wall rows completed from a saved
state) against the whole one.

Against the FP64 oracle the bar is the parity tests' 1e-5 per field (FP32
storage, velocity on the scale max(|u|, 0.01)); a split run must equal the
whole one bit for bit.
"""
import numpy as np
import pytest

import workloads as W
from oracle.solver import Oracle

pytestmark = pytest.mark.gpu

# 8 rows and 32 columns per block, 4 columns per block of the completion
SIZES = [(7, 7), (8, 8), (9, 9), (33, 11), (31, 16), (66, 17), (65, 25)]


@pytest.fixture(scope="module")
def HLBM():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_10751_gb300 as pkg
    pkg.build()
    from paper_2411_10751_gb300.solver import HLBM as cls
    return cls


def _case(kind, nx, ny, Pr):
    if kind == "couette":
        c = W.couette(nx=nx, ny=ny, Re=10.0, Pr=Pr, developed=True)
    else:
        c = W.rayleigh_benard(nx=nx, ny=ny, Ra=20.0, Pr=Pr, roll=0.005)
    # a variation along the walls, so that every column differs
    x = np.arange(nx) / nx
    c.theta = W.fp32(c.theta * (1.0 + 0.002 * np.sin(2 * np.pi * x)))
    c.u[0] = W.fp32(c.u[0] + 0.003 * np.cos(2 * np.pi * x))
    return c


@pytest.mark.parametrize("Pr", [1.0, 1.41])
@pytest.mark.parametrize("kind", ["couette", "benard"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_wall_step_at_block_edges(HLBM, kind, nx, ny, Pr):
    c = _case(kind, nx, ny, Pr)
    g = HLBM(c.lattice, nx, ny, 1, c.tau_hat, c.params)
    o = Oracle(c.lattice, nx, ny, 1, c.tau_hat, c.params)
    for s in (g, o):
        s.init(c.rho, c.u, c.theta)
    g.step(12)
    o.run(12)
    (rho, u, th), (r0, u0, t0) = g.moments_host(), o.moments()
    g.close()
    assert np.abs(rho - r0).max() / np.abs(r0).max() < 1e-5
    assert np.abs(th - t0).max() / np.abs(t0).max() < 1e-5
    assert np.sqrt(((u - u0) ** 2).sum(0)).max() / max(np.sqrt((u0 ** 2).sum(0)).max(), 0.01) < 1e-5


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("nx,ny", [(9, 7), (66, 17), (50, 56)])
def test_completion_in_the_step_equals_that_from_a_saved_state(HLBM, nx, ny, storage):
    c = _case("benard", nx, ny, 1.41)
    g = HLBM(c.lattice, nx, ny, 1, c.tau_hat, c.params, storage=storage)
    g.init(c.rho, c.u, c.theta)
    g.step(40)
    whole = g.save()
    g.init(c.rho, c.u, c.theta)
    g.step(33)
    part = g.save()
    g.step(3)          # other contents in the completion buffer
    g.load(part)
    g.step(7)
    assert g.save() == whole
    g.close()
