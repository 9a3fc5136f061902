"""The wait between the column passes of different warps, run as host threads under the thread
sanitizer (tests/wait_check.cpp): every lane's read of the rows is ordered after their writes."""
import os
import shutil
import subprocess

import pytest

from test_planner import CSRC, HERE, _cuda_include


@pytest.mark.skipif(shutil.which("g++") is None or _cuda_include() is None,
                    reason="no host C++ compiler or CUDA headers")
def test_every_lane_is_ordered_after_the_rows(tmp_path):
    exe = str(tmp_path / "wait_check")
    probe = subprocess.run(["g++", "-fsanitize=thread", "-x", "c++", "-", "-o", str(tmp_path / "p")],
                           input="int main() { return 0; }", text=True, capture_output=True)
    if probe.returncode != 0 or subprocess.run([str(tmp_path / "p")]).returncode != 0:
        pytest.skip("no thread sanitizer")
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-fsanitize=thread", "-I", CSRC, "-I",
                    _cuda_include(), os.path.join(HERE, "wait_check.cpp"), "-o", exe, "-pthread"],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr[-3000:]
