"""The fused embedding kernel at its tile edges: a tile holds two blocks of
128 rows, a block floor(129 / (L + 1)) words of one length L (at most 64).

Counts around one block and one tile, for the shortest and longest lengths,
mixed with an empty word.  A word's outputs do not depend on the words around
it (every output is the same sum in the same order), so the rows are equal bit
for bit to the same words embedded in another order among other lengths; and
they match the oracle's bf16 mode within the element-wise bound derived in
test_gpu_proposal.py.
"""
import numpy as np
import pytest

from oracle import proposal as PR
from paper_2509_01654_gb300 import nw, synth

pytestmark = pytest.mark.gpu

RTOL = 2.0 ** -6  # a few bf16 units, see test_gpu_proposal.py


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2509_01654_gb300 import build
    build.build()
    c = nw.Context(0)
    yield c
    c.close()


def words_per_block(L):
    return min(64, 129 // (L + 1))


@pytest.mark.parametrize("L", [0, 1, 2, 7, 15, 31, 39, 40])
def test_embedding_at_block_and_tile_edges(ctx, L):
    b = words_per_block(L)
    m = nw.Model(ctx, 40, seed=7)
    flat = np.random.default_rng(11).normal(0.0, 0.15, PR.param_count(40)).astype(np.float32)
    m.set_params(flat)
    for n in sorted({1, max(1, b - 1), b, b + 1, 2 * b, 2 * b + 1}):
        w = synth.make_uniform_length_words(n, 40, 1.0, L, L, seed=100 * L + n)
        got = m.embed(ctx.load_dictionary(w.codes, w.offsets, 40, (1, -1, -1)))
        # the same words, reversed, behind words of all lengths
        pad = synth.make_uniform_length_words(61, 40, 1.0, 0, 40, seed=n)
        lists = [pad.word(i) for i in range(pad.n)] + [w.word(i) for i in range(n)][::-1]
        codes = np.concatenate([np.asarray(x, dtype=np.uint8) for x in lists] + [np.zeros(0, np.uint8)])
        offs = np.concatenate([[0], np.cumsum([len(x) for x in lists])]).astype(w.offsets.dtype)
        mixed = m.embed(ctx.load_dictionary(codes, offs, 40, (1, -1, -1)))
        assert np.array_equal(got, mixed[pad.n:][::-1]), (L, n)
        want = PR.forward(flat.astype(np.float64), w, 40, bf16=True)
        atol = RTOL * float(np.sqrt(np.mean(want * want)))
        assert (np.abs(got - want) <= atol + RTOL * np.abs(want)).all(), (L, n)
