"""Host check of the workspaces that the library owns (no GPU): compiles
tests/native/workspace_check.cpp, which stands in for the CUDA runtime, against
csrc/workspace.h and runs it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(CUDA_INCLUDE), reason="needs g++ and CUDA headers")
def test_workspaces(tmp_path):
    exe = tmp_path / "workspace_check"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CUDA_INCLUDE, "-o", str(exe),
                    os.path.join(HERE, "native", "workspace_check.cpp")], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
