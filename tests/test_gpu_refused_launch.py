"""A launch that the driver refuses (a grid of more than 65,535 tile rows) fails its own
context and nothing else: a context made afterwards steps as ever.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,lag", [(7, False), (8, True)])   # the direct and the in-place step
def test_refused_launch_stays_with_its_context(nx, lag):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_10751_gb300 as pkg
    pkg.build()
    from paper_2411_10751_gb300 import abi
    from paper_2411_10751_gb300.solver import HLBM
    ny = 65536 * 8
    p = W.source_params(lag=True) if lag else W.source_params()
    one, u = np.ones((ny, nx), np.float32), np.zeros((2, ny, nx), np.float32)
    bad = HLBM("D2Q37", nx, ny, 1, 0.8, p, storage="f16")
    bad.init(one, u, one)
    with pytest.raises(abi.HLBMError) as e:
        bad.step(1)
    assert e.value.status == abi.HLBM_ECUDA
    c = W.kolmogorov(32)
    good = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params)
    good.init(c.rho, c.u, c.theta)
    good.step(3)
    good.synchronize()
    assert np.isfinite(good.diag()).all()
    good.close()
    bad.close()
