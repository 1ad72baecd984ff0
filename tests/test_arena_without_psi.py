"""A pseudopotential context's psi field serves one form of its step only.  Memory without
room for it is bound as well, and the step's results do not depend on it.
"""
import ctypes as C

import numpy as np
import pytest

import workloads as W


def _sizes(abi, c, storage):
    from paper_2411_10751_gb300.solver import make_params
    p = make_params(c.params, storage)
    total = abi.hlbm_workspace_bytes(0, c.nx, c.ny, 1, C.byref(p))
    psi = 0 if c.params.get("lag") else (4 * c.nx * c.ny + 255) // 256 * 256
    return p, total, total - psi


@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("lag", [False, True])
def test_bound_size_limit(storage, lag):
    from paper_2411_10751_gb300 import abi
    c = W.droplet(n=64, r0=16.0)
    c.params = dict(c.params, lag=lag)
    p, total, least = _sizes(abi, c, storage)
    for size, status in ((least, abi.HLBM_OK), (least - 1, abi.HLBM_ENOMEM), (total, abi.HLBM_OK)):
        ctx = C.c_void_p()
        assert abi.hlbm_create(0, c.nx, c.ny, 1, c.tau_hat, C.byref(p), C.byref(ctx)) == abi.HLBM_OK
        assert abi.hlbm_bind_memory(ctx, C.c_void_p(1 << 20), size) == status    # (not touched before hlbm_init)
        abi.hlbm_destroy(ctx)


@pytest.mark.gpu
@pytest.mark.parametrize("storage,nx,ny", [("f32", 512, 512), ("f16", 331, 403), ("f32", 64, 64)])
def test_step_without_room_for_psi(storage, nx, ny):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_10751_gb300 as pkg
    pkg.build()
    from paper_2411_10751_gb300 import abi
    from paper_2411_10751_gb300.solver import HLBM
    c = W.droplet(nx=nx, ny=ny, r0=0.25 * min(nx, ny), Tr=0.9)
    g = HLBM("D2Q37", nx, ny, 1, c.tau_hat, c.params, storage=storage)
    g.init(c.rho, c.u, c.theta)
    g.step(35)
    want = np.frombuffer(g.save(), np.uint8)
    g.close()
    p, total, least = _sizes(abi, c, storage)
    # the rest of the block stands for what the caller keeps behind the arena
    block = torch.full((total,), 0x5A, dtype=torch.uint8, device="cuda")
    ctx = C.c_void_p()
    abi.check(abi.hlbm_create(0, nx, ny, 1, c.tau_hat, C.byref(p), C.byref(ctx)))
    try:
        abi.check(abi.hlbm_bind_memory(ctx, C.c_void_p(block.data_ptr()), least), ctx)
        rho, u, th = (np.ascontiguousarray(a, dtype=np.float32) for a in (c.rho, c.u, c.theta))
        abi.check(abi.hlbm_init(ctx, rho.ctypes.data, u.ctypes.data, th.ctypes.data, 0), ctx)
        abi.check(abi.hlbm_step(ctx, 35), ctx)
        n = abi.hlbm_state_bytes(ctx)
        buf = C.create_string_buffer(n)
        abi.check(abi.hlbm_save(ctx, buf, n), ctx)
    finally:
        abi.hlbm_destroy(ctx)
    assert np.array_equal(np.frombuffer(buf.raw, np.uint8), want)
    assert (block[least:] == 0x5A).all()
