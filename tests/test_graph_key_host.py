"""Host check of the key of the library's CUDA-graph cache (no GPU): compiles
tests/native/graph_key_check.cpp against csrc/graph_key.h and runs it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(CUDA_INCLUDE), reason="needs g++ and CUDA headers")
def test_graph_key_tells_solves_apart(tmp_path):
    exe = tmp_path / "graph_key_check"
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CUDA_INCLUDE, "-o", str(exe),
                    os.path.join(HERE, "native", "graph_key_check.cpp")], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
