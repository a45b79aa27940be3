"""The fused backward kernel at its tile edges: a tile is 128 padded rows (every
non-empty word's rows and one zero row), and the batch may hold empty words, one
row, a row less or more than a tile, or more tiles than there are SMs.

Against the oracle's bf16 mode with the element-wise bound that
test_gpu_proposal.py derives for gradients (RTOL = 2^-6 of the element and of
the tensor's rms).
"""
import numpy as np
import pytest

from oracle import proposal as PR
from paper_2509_01654_gb300 import nw, synth

pytestmark = pytest.mark.gpu

RTOL = 2.0 ** -6


@pytest.fixture(scope="module")
def ctx():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2509_01654_gb300 import build
    build.build()
    c = nw.Context(0)
    yield c
    c.close()


# (shortest, longest word, pairs): padded rows 2 m (L + 1) for fixed lengths
@pytest.mark.parametrize("lo,hi,m,alphabet", [
    (0, 0, 5, 40),      # no row at all
    (1, 1, 1, 40),      # 4 padded rows
    (1, 1, 32, 40),     # 128: one full tile
    (31, 31, 2, 40),    # 128, the last row a zero row
    (40, 40, 3, 7),     # 246: words across the tile edge
    (42 - 2, 40, 25, 256),
    (0, 3, 333, 40),    # many empty words
    (0, 40, 700, 256),  # more tiles than SMs
])
def test_gradient_at_tile_edges(ctx, lo, hi, m, alphabet):
    w = synth.make_uniform_length_words(200, alphabet, 1.0, lo, hi, seed=lo + hi + m)
    d = ctx.load_dictionary(w.codes, w.offsets, alphabet, (1, -1, -1))
    model = nw.Model(ctx, alphabet, seed=5)
    flat = np.random.default_rng(23).normal(0.0, 0.15, PR.param_count(alphabet)).astype(np.float32)
    model.set_params(flat)
    g = np.random.default_rng(m)
    pi, pj = g.integers(0, w.n, m), g.integers(0, w.n, m)
    y = g.uniform(-1, 1, m).astype(np.float32)
    loss, grad = model.loss_grad(d, pi, pj, y)
    want_loss, want = PR.loss_and_grad(flat.astype(np.float64), w, alphabet, pi, pj, y, bf16=True)
    assert abs(loss - want_loss) <= RTOL * abs(want_loss)
    o = 0
    for name, shape in PR.param_shapes(alphabet):
        size = int(np.prod(shape))
        a, b = grad[o:o + size].astype(np.float64), want[o:o + size]
        atol = RTOL * float(np.sqrt(np.mean(b * b)))
        bad = np.abs(a - b) > atol + RTOL * np.abs(b)
        assert not bad.any(), (name, int(bad.sum()), size, float(np.abs(a - b).max()), atol)
        o += size
