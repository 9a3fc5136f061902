"""Alignment cells at the wavefront's edges: one residue, the 4 positions of a step, the 32 lanes,
strips of 256 positions and one more, several strips, and ties: repeats of a short motif, where
many cells reach the optimum and the first in row-major order counts, in either direction.  Both
entry points must equal the oracle's cells."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4, 8, 31, 33, 255, 256, 257, 300, 512, 513, 1025, 2100])
@pytest.mark.parametrize("kind", ["random", "motif", "one"])
def test_cells_match_oracle(n, kind):
    import torch
    rng = np.random.default_rng(n)
    motif = synth.random_seq(rng, 7)
    seqs = []
    for length in (n, 5, 130, 600):
        if kind == "random":
            seqs.append(synth.random_seq(rng, length))
        elif kind == "motif":
            seqs.append(np.resize(motif, length))
        else:
            seqs.append(np.full(length, 3, np.uint8))
    seqs.append(np.zeros(0, np.uint8))
    ss = synth.SeqSet.from_list(seqs)
    pairs = np.array([(0, k) for k in range(5)] + [(k, 0) for k in range(5)], np.int32)
    want = np.array([oracle.sw_cells(ss[x], ss[y], synth.BLOSUM62, 11, 1) for x, y in pairs])
    got = cm.sw_cells_batch(ss.seqs, ss.offsets, pairs, synth.BLOSUM62, 11, 1)
    assert np.array_equal(got, want)
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (ss.seqs, ss.offsets, pairs)]
    out = torch.full((len(pairs), 5), -7, dtype=torch.int32, device="cuda")
    cm.sw_cells_batch_noalloc(*dev, synth.BLOSUM62, 11, 1, out)
    assert np.array_equal(out.cpu().numpy(), want)
