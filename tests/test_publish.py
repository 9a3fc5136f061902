"""When the column passes of an alignment publish their boundary rows (csrc/cm_internal.h): on the
CPU the rule itself, on the GPU spans of several passes whose row groups end one after a multiple
of 32, where the step that ends the pass is also one that publishes."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth
from test_planner import CSRC, HERE, _cuda_include


@pytest.mark.skipif(shutil.which("g++") is None or _cuda_include() is None,
                    reason="no host C++ compiler or CUDA headers")
def test_last_group_is_never_published_in_the_loop(tmp_path):
    exe = str(tmp_path / "publish_check")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, "-I",
                    _cuda_include(), os.path.join(HERE, "publish_check.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


@pytest.mark.gpu
@pytest.mark.parametrize("rows,insert", [(n, 200) for n in range(128, 134)] +
                         [(n, 300) for n in range(256, 262)])
def test_spans_of_several_passes_match_oracle(rows, insert):
    rng = np.random.default_rng(rows)
    a = synth.random_seq(rng, rows)
    b = np.concatenate([a[:rows // 2], synth.random_seq(rng, insert), a[rows // 2:]])
    ss = synth.SeqSet.from_list([a, b])
    cells, offs, runs = cm.default_context().sw_align_batch(ss.seqs, ss.offsets,
                                                            np.array([(0, 1)] * 40, np.int32),
                                                            synth.BLOSUM62, 11, 1)
    want, ops = oracle.sw_align(ss[0], ss[1], synth.BLOSUM62, 11, 1)
    assert want[2] - want[1] + 1 == rows and want[4] - want[3] + 1 > 256
    for k in range(len(offs) - 1):
        assert tuple(cells[k]) == want
        assert [(int(v) >> 2, "MID"[int(v) & 3]) for v in runs[offs[k]:offs[k + 1]]] == ops
