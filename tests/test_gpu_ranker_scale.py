"""Ranker vectors of weights of any scale.  The logits are a cosine and the rectified layers are
homogeneous, so weights may be scaled freely: the first two layers up or down by a power of two and
the third back by it give the same network, whose activations differ by that power in every
rounding.  So the vectors must be the same to the bit, for short and long sequences; and those of
the plain weights are within BF16's rounding of the float64 oracle (3e-2 of the norm, as in
test_gpu_ranker_edges.py)."""
import numpy as np
import pytest

import paper_1908_10574_gb300 as cm
from oracle import ranker as R
from paper_1908_10574_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first,second", [(20, 10), (40, 0), (-20, -20), (-30, -40), (60, 30)])
def test_vectors_do_not_depend_on_the_scale_of_the_layers(first, second):
    rng = np.random.default_rng(2)
    ss = synth.SeqSet.from_list([synth.random_seq(rng, n) for n in (1, 3, 9, 40, 300, 5000, 0, 129)])
    flat = R.init_params(4).astype(np.float32)
    ctx = cm.Context(0)
    ctx.ranker_set_params(flat)
    plain = ctx.ranker_embed(ss.seqs, ss.offsets)
    want = R.embed(ss.seqs, ss.offsets, flat.astype(np.float64))
    for i in range(len(ss)):
        assert np.linalg.norm(plain[i] - want[i]) <= 3e-2 * np.linalg.norm(want[i])
    p = R.unpack(flat)                             # views into flat
    p["W1"] *= np.float32(2.0 ** first)
    p["b1"] *= np.float32(2.0 ** first)
    p["W2"] *= np.float32(2.0 ** second)
    p["b2"] *= np.float32(2.0 ** (first + second))
    p["W3"] *= np.float32(2.0 ** -(first + second))
    assert not np.array_equal(flat, R.init_params(4).astype(np.float32))
    ctx.ranker_set_params(flat)
    assert np.array_equal(ctx.ranker_embed(ss.seqs, ss.offsets), plain)


def test_vectors_follow_the_weights_of_training():
    """The scale belongs to the weights: after a training call and after new weights on the same
    context the vectors equal those of a new context with these weights."""
    rng = np.random.default_rng(6)
    ss = synth.SeqSet.from_list([synth.random_seq(rng, n) for n in (30, 31, 200, 64)])
    ctx = cm.Context(0)
    flat = R.init_params(8).astype(np.float32)
    ctx.ranker_set_params(flat)
    ctx.ranker_embed(ss.seqs, ss.offsets)
    pairs = np.array([(0, 1), (2, 3)], np.int32)
    ctx.ranker_train(ss.seqs, ss.offsets, pairs, np.array([1.0, 0.0], np.float32), epochs=40,
                     batch_pairs=2, lr=0.5)
    for _ in range(2):
        got = ctx.ranker_embed(ss.seqs, ss.offsets)
        now = ctx.ranker_get_params()
        new = cm.Context(0)
        new.ranker_set_params(now)
        assert np.array_equal(got, new.ranker_embed(ss.seqs, ss.offsets))
        p = R.unpack(now)
        p["W2"] *= np.float32(2.0 ** 30)
        p["b2"] *= np.float32(2.0 ** 30)
        p["W3"] *= np.float32(2.0 ** -30)
        ctx.ranker_set_params(now)
