"""Runs of the kernels that a context takes by size, for the bounds-checked debug build
(as debug_cases.py, whose cases are too small for them):

    HLBM_LIBRARY=debug python tests/debug_cases_large.py out.npz
"""
from __future__ import annotations

import sys
from pathlib import Path

sys.path.insert(0, str(Path(__file__).resolve().parent))

import debug_cases as D  # noqa: E402
import workloads as W  # noqa: E402


def cases():
    """name -> callable(solver module) returning a list of arrays."""
    def in_place_staged_even(S):        # boxes of the one buffer, steps of both parities
        return D._run(S.HLBM, D._lagged(W.thermal_decay(nx=1024, ny=640)), 4)

    def in_place_staged_odd(S):         # ragged tiles beside boxed ones
        return D._run(S.HLBM, D._lagged(W.thermal_decay(nx=900, ny=741)), 3)

    def in_place_staged_droplet(S):
        return D._run(S.HLBM, D._lagged(W.droplet(nx=1024, ny=640, r0=150.0)), 5)

    def in_place_staged_body_force(S):
        c = W.kolmogorov(nx=1024, ny=716, g0=1e-4)
        c.gfield = c.gfield[:, :, 0].copy()
        return D._run(S.HLBM, D._lagged(c), 5, field_kind="profile")

    def droplet_two_launches(S):        # psi of every node, then the step that reads it
        return D._run(S.HLBM, W.droplet(n=352, r0=80.0), 8)

    def droplet_two_launches_unaligned_f16(S):
        return D._run(S.HLBM, W.droplet(nx=331, ny=403, r0=80.0), 8, storage="f16")

    def thermal_direct_beyond_a_wave(S):
        return D._run(S.HLBM, W.thermal_decay(nx=331, ny=403), 8, storage="bf16")

    def thermal_ragged_one_cta_per_tile(S):   # edge tiles, ragged rows and columns, TMA stores
        return D._run(S.HLBM, W.thermal_decay(nx=200, ny=122), 12, (8, 2, 1))

    def thermal_persistent_default(S):
        return D._run(S.HLBM, W.thermal_decay(nx=648, ny=520), 8)

    return {k: v for k, v in locals().items() if callable(v)}


if __name__ == "__main__":
    D.cases = cases
    D.main(sys.argv[1])
