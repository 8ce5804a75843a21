"""FP32 thresholds take the FP64 light and lobe decisions exactly (host build
of the function that the scene builder and the table kernels share)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


@pytest.mark.parametrize("opt", ["-O0", "-O2"])
def test_unit_threshold_equals_fp64_decision(tmp_path, opt):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "threshold_check")
    subprocess.run([gxx, opt, "-std=c++17", "-I", os.path.join(ROOT, "paper_1903_07145_gb300", "csrc"), "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "threshold_check.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
