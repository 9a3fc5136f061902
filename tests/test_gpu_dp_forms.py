"""The packed cell update at the scoring schemes where a 16-bit half could carry into the other:
matrices down to -128 and up to 127, gaps below the least
score, free extensions, scores that leave int16 in one half only, 20 and 24 letters, through pair
lists (one query per warp) and the all-against-all (query pairs).  Scores are integers and must
equal the oracle's."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


def _matrix(lo, hi, alphabet):
    rng = np.random.default_rng(1000 + lo + hi)
    m = rng.integers(lo, hi + 1, size=(alphabet, alphabet))
    m = np.triu(m) + np.triu(m, 1).T
    m[0, 1] = m[1, 0] = lo
    m[np.arange(alphabet), np.arange(alphabet)] = hi
    return m.astype(np.int8)


@pytest.mark.parametrize("lo,hi,gap,ext", [
    (-4, 11, 11, 1),
    (-12, 11, 11, 1),           # least score below the gap
    (-11, 116, 11, 11),         # identical pairs leave int16
    (-128, 127, 1, 0),          # the widest matrix, free extensions
    (-128, 127, 1000, 1000),
    (-128, -1, 5, 1),           # no positive score
    (0, 9, 127, 0),
    (0, 0, 1, 1),
])
@pytest.mark.parametrize("alphabet", [20, 24])
def test_scoring_schemes_match_oracle(lo, hi, gap, ext, alphabet):
    rng = np.random.default_rng(7)
    root = rng.integers(0, alphabet, size=620).astype(np.uint8)
    seqs = []
    for n in [1, 4, 17, 40, 255, 256, 257, 500, 513, 600] * 9:
        s = root[:n].copy()
        hit = rng.random(n) < rng.choice([0.0, 0.3, 0.9])
        s[hit] = rng.integers(0, alphabet, size=int(hit.sum()))
        seqs.append(s)
    ss = synth.SeqSet.from_list(seqs)
    S = _matrix(lo, hi, alphabet)
    pairs = np.array([(i, j) for j in range(len(ss)) for i in range(j)], np.int32)
    want = oracle.sw_batch(ss.seqs, ss.offsets, pairs, S, gap, ext)
    ctx = cm.Context(0)
    some = rng.permutation(len(pairs))[:700]
    got = ctx.sw_score_batch(ss.seqs, ss.offsets, pairs[some], S, gap, ext)
    assert np.array_equal(got, want[some])
    keep = want > 0
    truth = sorted(zip(pairs[keep, 0].tolist(), pairs[keep, 1].tolist(), want[keep].tolist()))
    for warps in (16, 4):                     # all tiles in one launch, and a launch per tile
        ctx.set_tuning(warps, 0)
        p, s = ctx.sw_allpairs(ss.seqs, ss.offsets, S, gap, ext, 0)
        assert sorted(zip(p[:, 0].tolist(), p[:, 1].tolist(), s.tolist())) == truth
