"""The kernel of alignment cells whose scores may reach 2^28, which only pairs of more than two
million residues each reach through the library: run by itself on ordinary pairs
(tests/huge_cells_check.cu)."""
import os
import shutil
import subprocess

import pytest

from test_planner import CSRC, HERE

pytestmark = pytest.mark.gpu


def test_huge_score_kernel_matches_the_recurrences(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "huge_cells_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC,
                    os.path.join(HERE, "huge_cells_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout + out.stderr
