"""A learned ClusterMerge whose device-built lists put a run of long subjects into one task of a lone
query of four passes (the lists are cut by count): the task's streams are longer than the boundary
slot of its warp, so it runs in pieces.  Nothing is pruned, so clusters and pairs must equal the
oracle's."""
import numpy as np
import pytest

import oracle
import paper_1908_10574_gb300 as cm
from oracle import ranker as R
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu
S62 = synth.BLOSUM62


def test_ranked_merge_of_a_run_of_long_subjects():
    rng = np.random.default_rng(17)
    domain = synth.random_seq(rng, 300)

    def long(n):                                   # a mutated domain somewhere in a random rest
        s = synth.random_seq(rng, n)
        at = int(rng.integers(0, n - 300))
        hit = rng.random(300) < 0.3
        s[at:at + 300] = np.where(hit, synth.random_seq(rng, 300), domain)
        return s

    seqs = [long(1990), long(1950)] + [synth.random_seq(rng, int(n)) for n in rng.integers(40, 60, 126)]
    seqs[100] = seqs[101].copy()                   # they merge: an odd number of queries, the longest alone
    seqs += [synth.random_seq(rng, int(n)) for n in rng.integers(40, 60, 108)]
    seqs += [long(int(n)) for n in rng.integers(1900, 2000, 20)]
    ss = synth.SeqSet.from_list(seqs)
    n = len(ss)
    _, scores = oracle.all_pairs(ss.seqs, ss.offsets, S62, 11, 1, T=100)
    M = np.zeros((n, n), np.int64)
    M[np.triu_indices(n, 1)] = scores
    M = M + M.T
    want = oracle.cluster_merge(ss.seqs, ss.offsets, S62, 11, 1, T=100, mT=138, mU=15, score_matrix=M)
    ctx = cm.Context(0)
    ctx.ranker_set_params(R.init_params(5).astype(np.float32))
    ctx.set_tuning(16, 256)
    got = ctx.cluster_merge(ss.seqs, ss.offsets, S62, 11, 1, 100, 138, 15, use_ranker=True,
                            prune_logit=-1e30, ranker_min_pairs=1)
    assert got["clusters"] == want["clusters"]
    assert got["pairs"].tolist() == want["pairs"].tolist()
