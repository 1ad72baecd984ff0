"""Registers of the staged D2Q37 step, as the assembler reports them: the 8-row
one-node schedules are sized for 80 registers (128 with the psi frame), and their
gather of an edge tile must fit beside the staged tile without spilling.
"""
import importlib
import re
import shutil
import subprocess

import pytest

SOURCE = """#include "step2d.cuh"
#define ARGS const __grid_constant__ StepArgs, const __grid_constant__ CUtensorMap, const __grid_constant__ CUtensorMap
namespace hlbm {
template __global__ void step2d_kernel<ST_F32, KIND_THERMAL, false, 8, 1>(ARGS);
template __global__ void step2d_persistent_kernel<ST_F32, KIND_THERMAL, 8, 1>(ARGS);
template __global__ void step2d_persistent_kernel<ST_F32, KIND_SC, 8, 1>(ARGS);
}
"""


def test_one_node_staged_kernels_do_not_spill(tmp_path):
    B = importlib.import_module("paper_2411_10751_gb300.build")
    if shutil.which(B.NVCC) is None:
        pytest.skip("no nvcc")
    if not (B.BUILD / "lattice_weights.inc").exists():
        B.build()
    (tmp_path / "k.cu").write_text(SOURCE)
    r = subprocess.run([B.NVCC, *B.ARCH, *B.CFLAGS, "-Xptxas", "-v", "-c", str(tmp_path / "k.cu"), "-o",
                        str(tmp_path / "k.o")], capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-2000:]
    spills = [int(n) for n in re.findall(r"(\d+) bytes spill stores", r.stderr)]
    assert spills == [0, 0, 0], r.stderr
