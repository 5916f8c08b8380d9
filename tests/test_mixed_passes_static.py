"""Host-only check (no GPU): the mixed plans' passes, templates over the real
type with FP32 tables and copies inside, do not compile for FP64."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("real,ok", [("float", True), ("double", False)])
def test_inverse_row_pass(tmp_path, real, ok):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "inst.cu"
    src.write_text('#include "kernels.cuh"\n'
                   f"template __global__ void dsnu::k_row_inv<{real}, 4>(dsnu::Members, dsnu::WsOff, int, int, int, int, "
                   f"dsnu::AxisTabs<{real}>, const {real}*, {real}, int, int, int);\n")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                        "-I" + os.path.join(ROOT, "paper_1409_2014_gb300", "csrc"), "-I" + os.path.join(ROOT, "include"),
                        "-c", str(src), "-o", str(tmp_path / "inst.o")], capture_output=True, text=True)
    assert (r.returncode == 0) == ok, r.stderr
    assert ok or "static assertion failed" in r.stderr
