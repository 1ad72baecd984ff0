"""The D2Q37 step without staging (contexts without a schedule) against the
staged one (one CTA per tile, two nodes per thread): bit for bit, at the edges of
its tiles, on rows of every 16-byte remainder, on domains narrower than a tile's
frame, around one wave of blocks, and with every kind of body force.
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


def _case(kind, nx, ny):
    if kind == "thermal":
        return W.thermal_decay(nx=nx, ny=ny, tau_hat=0.7, Pr=0.71)
    if kind == "thermal_forced":
        c = W.kolmogorov(nx=nx, ny=ny, g0=1e-4)
        c.params.update(H=True, Pr=0.9)
        c.theta = W.fp32(c.theta + 0.01 * np.sin(2 * np.pi * np.arange(nx) / nx))
        return c
    if kind == "kolmogorov":
        return W.kolmogorov(nx=nx, ny=ny, g0=1e-4)
    eos = "cs" if kind == "cs_droplet" else "vdw"
    return W.droplet(nx=nx, ny=ny, r0=0.25 * min(nx, ny), Tr=0.9, k=3.02 if eos == "cs" else 1.5672, eos=eos)


def _run(HLBM, c, storage, schedule, force_kind, steps):
    g = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params, storage=storage)
    if schedule:
        g.set_tile(*schedule)
    if c.gfield is not None:
        g.set_force_field(c.gfield[:, :, 0] if force_kind == "profile" else c.gfield, force_kind)
    g.init(c.rho, c.u, c.theta)
    g.step(steps)
    s = g.save()
    g.close()
    return s


# 7 x 7 and 9 x 40: narrower than the frame; 32 x 8: one tile; 31 .. 35: the
# remainders of a tile; 157 x 151: tiles around the SM count and odd rows;
# 219 x 300, 288 x 290: several waves of blocks, rows off and on the 16-byte grid
SIZES = [(7, 7), (9, 40), (32, 8), (33, 9), (34, 15), (35, 17), (64, 64), (157, 151), (219, 300), (288, 290)]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind", ["kolmogorov", "thermal", "thermal_forced", "droplet", "cs_droplet"])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_direct_step_equals_staged(HLBM, kind, nx, ny, storage):
    c = _case(kind, nx, ny)
    for force_kind in ("profile", "field") if c.gfield is not None else (None,):
        a = _run(HLBM, c, storage, None, force_kind, 5)
        b = _run(HLBM, c, storage, (8, 2, 1), force_kind, 5)
        assert a == b
