"""Query pairs of many register tiles in one launch (plans too small to fill the chip tile by
tile): the all-against-all of sets whose lengths sit at the tiles' edges, in 16-lane segments, over
32 lanes and in several column passes, whole and in parts, must equal the oracle's; and the
default launch must equal the launch per tile that a narrower CTA takes."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


def _set(lengths, alphabet):
    rng = np.random.default_rng(len(lengths) + alphabet)
    root = rng.integers(0, alphabet, size=max(lengths)).astype(np.uint8)
    seqs = []
    for n in lengths:
        s = root[:n].copy()
        hit = rng.random(n) < 0.5
        s[hit] = rng.integers(0, alphabet, size=int(hit.sum()))
        seqs.append(s)
    return synth.SeqSet.from_list(seqs)


@pytest.mark.parametrize("lengths", [
    [1, 2, 3, 15, 16, 17, 31, 32, 33] * 12,                     # narrow 16-lane tiles
    [255, 256, 257, 496, 497, 511, 512, 513, 544, 545] * 8,     # both lane counts
    [40] * 70 + [1023, 1024, 1025, 1030, 2047, 2049],           # passes over many subjects
])
@pytest.mark.parametrize("parts", [1, 3])
@pytest.mark.parametrize("alphabet", [20, 24])
def test_all_pairs_match_oracle(lengths, parts, alphabet):
    ss = _set(lengths, alphabet)
    S = synth.BLOSUM62 if alphabet == 20 else synth.BLOSUM62_24
    pairs = np.array([(i, j) for j in range(len(ss)) for i in range(j)], np.int32)
    want = oracle.sw_batch(ss.seqs, ss.offsets, pairs, S, 11, 1)
    keep = want > 20
    truth = sorted(zip(pairs[keep, 0].tolist(), pairs[keep, 1].tolist(), want[keep].tolist()))
    for warps in (16, 4):
        ctx = cm.Context(0)
        ctx.set_tuning(warps, 0)
        got = []
        for part in range(parts):
            p, s = ctx.sw_allpairs(ss.seqs, ss.offsets, S, 11, 1, 20, part, parts)
            got += list(zip(p[:, 0].tolist(), p[:, 1].tolist(), s.tolist()))
        assert sorted(got) == truth
