"""Pair lists whose lone queries have several column passes and more units of work than the chip has
warps, so that every range of the launch holds tasks behind one another; and fewer tasks than CTAs,
so that CTAs share ranges.  Scores are integers and must equal the oracle's."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("queries,longest", [(900, 1600), (5, 6000)])
def test_units_of_many_pipelined_tasks(queries, longest):
    rng = np.random.default_rng(queries)
    root = synth.random_seq(rng, longest)
    seqs = []
    for n in np.concatenate([rng.integers(513, longest + 1, size=queries), rng.integers(1, 400, size=40)]):
        s = root[:n].copy()
        hit = rng.random(n) < 0.5
        s[hit] = synth.random_seq(rng, int(hit.sum()))
        seqs.append(s)
    ss = synth.SeqSet.from_list(seqs)
    pairs = np.array([(q, queries + int(s)) for q in range(queries) for s in rng.integers(0, 40, size=3)],
                     np.int32)
    want = oracle.sw_batch(ss.seqs, ss.offsets, pairs, synth.BLOSUM62, 11, 1)
    assert np.array_equal(cm.Context(0).sw_score_batch(ss.seqs, ss.offsets, pairs, synth.BLOSUM62, 11, 1), want)
