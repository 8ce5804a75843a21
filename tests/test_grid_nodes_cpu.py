"""The scene-grid 4-wide nodes on the host (tests/grid_check.cpp, compiled with
the scene builder): same tree as the 8-bit nodes, boxes that hold their
triangles, no exact hit missed by the traversal's plane arithmetic, and the
scenes that keep the 8-bit nodes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_scene_grid_nodes(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path / "grid_check")
    csrc = os.path.join(ROOT, "paper_1903_07145_gb300", "csrc")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", csrc,
                    "-I", CUDA_INC, os.path.join(ROOT, "tests", "grid_check.cpp"),
                    os.path.join(csrc, "scene_build.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
