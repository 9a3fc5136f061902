"""Alignments whose spans end at the traceback kernel's edges: one residue, the 8 columns of a
lane, the 4 rows of a step, the 256 columns of a pass and one more, several passes; equal
sequences and ones with a block inserted or deleted, so that the walk crosses lanes, passes and
long gaps.  Cells and every run must equal the oracle's."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 5, 8, 9, 128, 255, 256, 257, 512, 513, 1100])
@pytest.mark.parametrize("gap", [0, 1, 40])
def test_span_edges_match_oracle(n, gap):
    rng = np.random.default_rng(100 * n + gap)
    a = synth.random_seq(rng, n)
    b = np.concatenate([a[:n // 2], synth.random_seq(rng, gap), a[n // 2:]])
    ss = synth.SeqSet.from_list([a, b])
    pairs = np.array([(0, 0), (0, 1), (1, 0)], np.int32)
    ctx = cm.default_context()
    cells, offs, runs = ctx.sw_align_batch(ss.seqs, ss.offsets, pairs, synth.BLOSUM62, 11, 1)
    for k, (x, y) in enumerate(pairs):
        want, ops = oracle.sw_align(ss[x], ss[y], synth.BLOSUM62, 11, 1)
        assert tuple(cells[k]) == want
        assert [(int(v) >> 2, "MID"[int(v) & 3]) for v in runs[offs[k]:offs[k + 1]]] == ops
