"""The one-warp kernel of lone queries (sw_score_batch's pair lists) at the sizes where it can go
wrong: tile and pass edges, queries whose column passes run as a pipeline of warps, streams with
no subject, one subject only, empty sequences, an asymmetric 24-letter matrix; and the int32
rescoring of the same pairs.  Scores are integers and must equal the oracle's."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return cm.Context(0)


@pytest.mark.parametrize("queries,subjects", [
    ([1, 15, 16, 17, 255, 256], [1]),                       # 16-lane tiles, one subject
    ([257, 288, 289, 511, 512], [0, 1, 3, 4, 5, 700]),      # one pass of 32 lanes
    ([513, 1024, 1025, 1536], [1, 130, 513, 2047]),         # two and three passes, pipelined
    ([2900, 5000], [5000, 4, 2900, 128, 124, 0]),           # many passes, uneven streams
])
@pytest.mark.parametrize("alphabet", [20, 24])
def test_pair_lists_match_oracle(ctx, queries, subjects, alphabet):
    rng = np.random.default_rng(sum(queries) + alphabet)
    root = rng.integers(0, alphabet, size=max(queries + subjects)).astype(np.uint8)
    seqs = []
    for n in queries + subjects:                            # related, so scores grow with length
        s = root[:n].copy()
        hit = rng.random(n) < 0.4
        s[hit] = rng.integers(0, alphabet, size=int(hit.sum()))
        seqs.append(s)
    ss = synth.SeqSet.from_list(seqs)
    nq = len(queries)
    pairs = np.array([(q, nq + s) for q in range(nq) for s in range(len(subjects))] +
                     [(nq + s, q) for s in range(len(subjects)) for q in range(nq)], np.int32)
    S = synth.BLOSUM62 if alphabet == 20 else rng.integers(-9, 10, size=(24, 24)).astype(np.int8)
    want = oracle.sw_batch(ss.seqs, ss.offsets, pairs, S, 11, 1)
    assert np.array_equal(ctx.sw_score_batch(ss.seqs, ss.offsets, pairs, S, 11, 1), want)
    # the same pairs through the int32 strips
    assert np.array_equal(ctx.sw_score_batch(ss.seqs, ss.offsets, pairs, S, 11, 1,
                                             flags=cm.CM_FORCE_INT32), want)
