"""The D2Q37 step without staging on unaligned rows around and beyond one wave of its
blocks, against the staged step (one CTA per tile, two nodes per thread): bit for bit.
Beyond one wave the pseudopotential step is two launches (psi of every node, then the
step that reads it), in every storage.
"""
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
    if kind == "kolmogorov":
        return W.kolmogorov(nx=nx, ny=ny, g0=1e-4)
    eos = "cs" if kind == "cs_droplet" else "vdw"
    return W.droplet(nx=nx, ny=ny, r0=0.25 * min(nx, ny), Tr=0.9, k=3.02 if eos == "cs" else 1.5672, eos=eos)


def _run(HLBM, c, storage, schedule):
    g = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params, storage=storage)
    if schedule:
        g.set_tile(*schedule)
    if c.gfield is not None:
        g.set_force_field(c.gfield[:, :, 0], "profile")
    g.init(c.rho, c.u, c.theta)
    g.step(35)              # a graph of 32 steps, then single launches
    s = g.save()
    g.close()
    return s


# blocks per SM (step2d_direct.cuh): 2 thermal, 2 pseudopotential (1 while the tiles
# fit one per SM), 3 body force
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind", ["kolmogorov", "thermal", "droplet", "cs_droplet"])
@pytest.mark.parametrize("nx,ny,above,upto", [(230, 211, 1, 2), (331, 403, 3, 99), (641, 639, 3, 99)])
def test_direct_step_around_a_wave_of_blocks(HLBM, kind, nx, ny, above, upto, storage):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = ((nx + 31) // 32) * ((ny + 7) // 8)
    assert above * sms < tiles <= upto * sms
    assert nx * (4 if storage == "f32" else 2) % 16, "rows must be off the 16-byte grid"
    c = _case(kind, nx, ny)
    assert _run(HLBM, c, storage, None) == _run(HLBM, c, storage, (8, 2, 1))


@pytest.mark.parametrize("kind,nx,ny", [("thermal", 640, 520), ("droplet", 640, 520), ("droplet", 352, 344)])
def test_default_of_large_aligned_domains(HLBM, kind, nx, ny):
    """FP32: the persistent kernels (two buffers beyond 96 MB), and two launches below."""
    c = _case(kind, nx, ny)
    assert _run(HLBM, c, "f32", None) == _run(HLBM, c, "f32", (8, 2, 1))
