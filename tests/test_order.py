"""The counting sort that orders pair lists and alignment jobs (csrc/plan.h), without a GPU."""
import os
import shutil
import subprocess

import pytest

from test_planner import CSRC, HERE, _cuda_include


@pytest.mark.skipif(shutil.which("g++") is None or _cuda_include() is None,
                    reason="no host C++ compiler or CUDA headers")
def test_counting_order(tmp_path):
    exe = str(tmp_path / "order_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-I",
                    _cuda_include(), os.path.join(HERE, "order_check.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
