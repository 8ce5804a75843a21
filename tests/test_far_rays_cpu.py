"""Rays from far away and the empty slots of the 4-wide nodes on the host
(tests/far_rays_check.cpp, compiled with the scene builder)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_far_rays_enter_no_empty_slot(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "far_rays_check")
    csrc = os.path.join(ROOT, "paper_1903_07145_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", csrc,
                    "-I", CUDA_INC, os.path.join(ROOT, "tests", "far_rays_check.cpp"),
                    os.path.join(csrc, "scene_build.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
