"""Ranker vectors of sequences at the edges of the inference kernels: none, one to nine residues
(shorter than the convolution's reach), lengths around the 32 rows of an epilogue warp and the
128 rows of a tile, more sequences than a block of the pooling kernel takes, codes without an
embedding.  Against the float64 oracle within BF16's rounding: three layers of operands and
activations rounded to 2^-9 each, 3e-2 of the vector's norm as elsewhere."""
import numpy as np
import pytest

import paper_1908_10574_gb300 as cm
from oracle import ranker as R
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[1], [0, 1, 2, 3, 4, 5, 6, 7, 8, 9],
                                     [31, 32, 33, 27, 28, 29] * 3,
                                     [127, 128, 129, 119, 120, 124, 257, 1000]])
def test_vectors_match_oracle(lengths):
    rng = np.random.default_rng(len(lengths))
    ss = synth.SeqSet.from_list([synth.random_seq(rng, n) for n in lengths])
    p = R.init_params(3).astype(np.float32)
    ctx = cm.Context(0)
    ctx.ranker_set_params(p)
    got = ctx.ranker_embed(ss.seqs, ss.offsets)
    want = R.embed(ss.seqs, ss.offsets, p.astype(np.float64))
    for i in range(len(ss)):
        assert np.linalg.norm(got[i] - want[i]) <= 3e-2 * np.linalg.norm(want[i]), lengths[i]
