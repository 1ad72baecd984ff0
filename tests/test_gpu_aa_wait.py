"""The bounded wait of the in-place step's staged form: tiles whose barrier is armed but
never receives its copies (test hook) give up after the wall-time limit and report
HLBM_ETIMEOUT through the status word, in both parities; the device stays usable.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("odd", [False, True])
def test_expired_wait_of_the_staged_in_place_step_reports_timeout(monkeypatch, odd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2411_10751_gb300 as pkg
    pkg.build()
    from paper_2411_10751_gb300 import abi
    from paper_2411_10751_gb300.solver import HLBM
    c = W.thermal_decay(nx=1024, ny=640)
    c.params = dict(c.params, lag=True)
    plain = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params)
    plain.init(c.rho, c.u, c.theta)
    plain.step(1 if odd else 2)
    state = plain.save()                    # the parity that the next step has
    monkeypatch.setenv("HLBM_TEST_SKIP_TMA", "1")
    g = HLBM(c.lattice, c.nx, c.ny, 1, c.tau_hat, c.params)
    monkeypatch.delenv("HLBM_TEST_SKIP_TMA")
    abi.check(abi.hlbm_set_wait_timeout(g.ctx, 0.01), g.ctx)
    g.load(state)
    g.step(1)
    with pytest.raises(abi.HLBMError) as e:
        g.synchronize()
    assert e.value.status == abi.HLBM_ETIMEOUT
    g.close()
    plain.step(3)
    assert np.isfinite(plain.diag()).all()
    plain.close()
