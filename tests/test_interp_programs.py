"""Programs of the expression interpreter, without a GPU: random trees in which fields occur several
times are compiled to programs, the programs run step by step, and every value compared with the
tree's own (tests/interp_programs.cpp: integers, so the comparison is exact)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def programs(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if cxx is None or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    exe = str(tmp_path_factory.mktemp("interp") / "programs")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1710_09409_gb300", "csrc"),
                           "-I", os.path.join(cuda, "include"), os.path.join(HERE, "interp_programs.cpp"), "-o", exe])
    return exe


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_random_trees(programs, seed):
    r = subprocess.run([programs, "50000", str(seed)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok 50000 trees") and " 0 refused" in r.stdout
